// order.cu -- the order in which a rollout launch takes its samples.
//
// A warp's 32 rollouts advance in lock step, so a warp is only as fast as its
// lanes are alike: rollouts last 1.5 to 10 s, a launch of one generation lasts
// as long as every warp's slowest lane, and in a long launch the lanes reach
// their events (onset, breakpoints of r(D), the end) in different passes.
// Taking the samples by predicted length, longest first, gives every warp
// rollouts that start, turn and end together and leaves short ones for the
// tail.  Results do not depend on the order: a sample's arithmetic never
// depends on the lanes it shares a warp with.
//
// The prediction is a closed form in binary32 (coasting, then the braking that
// the caps allow at full command, delayed by the area the actuator's ramp
// loses, drag at a mean speed), 9 ms off the true length in the mean on the
// single-scenario workload; it decides nothing but the order.  Samples whose
// braking ends on the constant cap (saturated friction) come first: they last
// longest, and a warp of them alone needs no actuator once it is there; among
// samples of one length (bins of 1/256 of the horizon) those whose r(D) settles
// early come first, so that a warp's lanes settle together (4 bins of 0.25 s:
// 1-2 % on most workloads; 512 length bins alone, or 32-128 with 4-16 turn
// bins: slower).
//
// Two kernels before the rollouts: bin every position by (cap class, length,
// turn), then scatter the positions to their bins' ranges (a counting sort; the
// order inside a bin is free).  Per sample 56 B of columns read (64 B with a
// lead, 72 B with the TTC trigger), a 2-byte key and a 4-byte position written
// and read.
#include <algorithm>
#include <cmath>

#include "rollout_common.cuh"

namespace aeb {
namespace {

constexpr int kLenBins = 256;                 // over [0, horizon]
constexpr int kTurnBins = 4;                  // of kTurnBin seconds, the last open
constexpr float kTurnBin = 0.25f;
constexpr int kClasses = 3;                   // constant cap, axle line, uncapped demand
constexpr int kBins = kClasses * kLenBins * kTurnBins;
constexpr uint16_t kNoSample = 0xffff;        // a position no tile uses
constexpr int kOrderThreads = 256;
// Positions per thread of the scatter: few in a small launch, which waits for
// one block's chain (1e5: 13.4 -> 7 us), more where the blocks' scans of the
// counts add up.
constexpr int kScatterFew = 4, kScatterMany = 16;
constexpr uint32_t kScatterSmall = 1u << 19;
// Positions ordered at a time, and so the bound on the scratch (100 MB).  A
// longer launch runs in pieces; each piece's tail costs ~0.3 ms of ~40.
constexpr uint64_t kOrderMax = uint64_t(1) << 24;
constexpr uint64_t kNaturalMax = uint64_t(1) << 31;

// Binary32 copies of the model's constants.
struct OrderModel {
    float D, g, rho_a2, hl, beta, phi_f, thr, lat, t_max, lv0, lb, lts, lxs;
    int lumped, ttc, lead, moving;
};

// x cut to binary32 on the integer pipe (a conversion instruction runs on the
// binary64 unit, 64 cycles a warp): 0 below the normal range, the largest value
// above it.  Good enough for an order.
__device__ __forceinline__ float cut_f32(double x)
{
    const uint32_t hi = (uint32_t)__double2hiint(x), lo = (uint32_t)__double2loint(x);
    const uint32_t m = hi & 0x7fffffffu;
    uint32_t b = ((m - (896u << 20)) << 3) | (lo >> 29);
    b = m < (897u << 20) ? 0u : m >= (1151u << 20) ? 0x7f7fffffu : b;
    return __int_as_float((int)(b | (hi & 0x80000000u)));
}

struct Motion {  // coasting at -a0 until tb, then braking at -b
    float v0, a0, tb, v1, x1, b;
    __device__ float x(float t) const
    {
        if (t <= tb) return t * (v0 - 0.5f * a0 * t);
        const float s = t - tb;
        return x1 + s * (v1 - 0.5f * b * s);
    }
};

// Predicted seconds until the rollout ends, its cap class, and the time at
// which r(D) reaches its last piece.
__device__ __forceinline__ float predict(const OrderModel &M, const ParamsDev &P, const Row &row,
                                         int &cls, float &turn)
{
    auto f = [&](int j) { return cut_f32(__ldg(P.col[j] + row.p)); };
    const float v0 = f(kV0), mu = f(kMu), gs = f(kGs), tau = f(kTau);
    const float mh = mu * M.hl;
    float r = M.D, B = 0.0f;  // B: the demand at the last breakpoint below M.D
    cls = 2;
    if (M.lumped) {
        const float c = __fdividef(mu * M.g, 1.0f + mh);
        if (c < r) {
            r = B = c;
            cls = 0;
        }
    } else {
        const float mg = mu * M.g;
        const float im = __fdividef(1.0f, 1.0f - mh), ip = __fdividef(1.0f, 1.0f + mh);
        const float f0 = mg * M.phi_f * im, f1 = (1.0f - M.beta) * im;
        const float r0 = mg * (1.0f - M.phi_f) * ip, r1 = M.beta * ip;
        const float lf = f0 + f1 * M.D, lr = r0 + r1 * M.D;
        if (fminf(lf, lr) < r) {
            r = fminf(lf, lr);
            cls = 1;
            B = lf < lr ? __fdividef(f0, 1.0f - f1) : __fdividef(r0, 1.0f - r1);
        }
        if (mg <= r) {
            r = mg;
            cls = 0;
            B = fmaxf(mg, fmaxf(__fdividef(mg - f0, f1), __fdividef(mg - r0, r1)));
        }
    }
    r = fmaxf(r, 1e-3f);
    const float k = __fdividef(M.rho_a2 * f(kCd), f(kMass));
    const float a0 = gs + k * v0 * v0;
    // the ramp min(r, D (1 - exp(-t / tau))) as a step to r, delayed by the
    // area it loses
    const float w = fminf(fmaxf(1.0f - __fdividef(r, M.D), 1e-6f), 1.0f);
    const float te = tau * fmaxf(1.0f + __fdividef(M.D - r, r) * __logf(w), 0.0f);
    float td = f(kTdelay) + M.lat;
    const float d0 = M.lead ? f(kD0) : 0.0f;
    if (M.ttc) {  // coasting until the measured gap reaches thr times the closing speed
        const float lb = M.moving ? M.lb : 0.0f;
        const float thr = cut_f32(row.thr);
        const float c0 = v0 - M.lv0, C = f(kD0) + f(kNoise) - thr * c0;
        if (C > 0.0f) {
            const float A = 0.5f * (lb - a0), B = c0 + thr * (lb - a0);
            const float q = B * B + 4.0f * A * C;
            const float t = (q > 0.0f) ? __fdividef(2.0f * C, B + sqrtf(q)) : M.t_max;
            td += (t > 0.0f) ? fminf(t, M.t_max) : M.t_max;
        }
    }
    turn = td - tau * __logf(fminf(fmaxf(1.0f - __fdividef(B, M.D), 1e-3f), 1.0f));
    Motion m;
    m.v0 = v0;
    m.a0 = a0;
    m.tb = td + te;
    m.v1 = fmaxf(v0 - a0 * m.tb, 0.1f);
    m.x1 = m.tb * (v0 - 0.5f * a0 * m.tb);
    const float kv = k * m.v1 * m.v1, b = fmaxf(r + gs, 0.05f);
    const float ts = m.tb + __fdividef(m.v1, b + kv * (1.0f / 3.0f));
    m.b = b + 0.5f * kv;
    const float sb = __fdividef(m.v1 * m.v1, 2.0f * m.b);  // braking distance
    if (!M.lead) return ts;
    if (!M.moving) {
        const float d = d0 - m.x1;
        if (d < 0.0f) return __fdividef(d0, v0);
        if (sb < d) return ts;
        // drag over the part of the braking distance that is driven
        const float bc = b + kv * (1.0f - 0.5f * __fdividef(d, sb));
        return m.tb + __fdividef(2.0f * d, m.v1 + sqrtf(fmaxf(m.v1 * m.v1 - 2.0f * bc * d, 0.0f)));
    }
    // moving lead: the first sign change of the gap over twelve parts of the
    // time to stop
    const float te12 = fminf(ts, M.t_max) * (1.0f / 12.0f);
    float g0 = d0;
    for (int i = 1; i <= 12; ++i) {
        const float t = te12 * (float)i;
        const float xl = (M.lb > 0.0f && t >= M.lts) ? M.lxs : t * (M.lv0 - 0.5f * M.lb * t);
        const float g1 = d0 + xl - m.x(t);
        if (g1 <= 0.0f) return t - te12 * (1.0f - __fdividef(g0, g0 - g1));
        g0 = g1;
    }
    return ts;
}

// Pass 1: each position's bin and the bins' counts.
__global__ void __launch_bounds__(kOrderThreads)
k_order_keys(OrderModel M, ParamsDev P, WorkDev W, uint32_t positions,
             uint32_t *__restrict__ hist, uint16_t *__restrict__ keys)
{
    __shared__ uint32_t sh[kBins];
    for (int j = threadIdx.x; j < kBins; j += kOrderThreads) sh[j] = 0u;
    __syncthreads();
    const uint32_t step = gridDim.x * kOrderThreads;
    for (uint32_t p = blockIdx.x * kOrderThreads + threadIdx.x; p < positions; p += step) {
        uint16_t key = kNoSample;
        if (!W.tiles || p % W.tile < W.tiles[p / W.tile].count) {
            int cls;
            float turn;
            const float t = predict(M, P, row_of(W, p, (double)M.thr), cls, turn);
            // longest first; a NaN counts as no time at all
            int len = (t > 0.0f) ? (int)(fminf(t * __fdividef((float)kLenBins, M.t_max), 1e6f)) : 0;
            len = len < kLenBins ? len : kLenBins - 1;
            const int tb = (int)fminf(fmaxf(turn * (1.0f / kTurnBin), 0.0f), kTurnBins - 1.0f);
            key = (uint16_t)((cls * kLenBins + (kLenBins - 1 - len)) * kTurnBins + tb);
            atomicAdd(&sh[key], 1u);
        }
        keys[p] = key;
    }
    __syncthreads();
    for (int j = threadIdx.x; j < kBins; j += kOrderThreads)
        if (sh[j]) atomicAdd(&hist[j], sh[j]);
}

// Pass 2: positions to their bins' ranges.  Each block ranks its positions in
// shared memory and reserves one range per bin it holds.
template <int ITEMS>
__global__ void __launch_bounds__(kOrderThreads)
k_order_scatter(uint32_t positions, const uint32_t *__restrict__ hist,
                uint32_t *__restrict__ cursor, const uint16_t *__restrict__ keys,
                uint32_t *__restrict__ perm)
{
    constexpr int kPer = kBins / kOrderThreads;
    static_assert(kBins % kOrderThreads == 0, "whole bins per thread");
    __shared__ uint32_t cnt[kBins], base[kBins];
    __shared__ uint32_t part[kOrderThreads / 32];
    const int t = threadIdx.x;
    // exclusive scan of the bin counts
    uint32_t own[kPer], sum = 0;
#pragma unroll
    for (int j = 0; j < kPer; ++j) {
        own[j] = __ldg(hist + t * kPer + j);
        sum += own[j];
        cnt[t * kPer + j] = 0u;
    }
    uint32_t inc = sum;
    for (int m = 1; m < 32; m <<= 1) {
        const uint32_t o = __shfl_up_sync(kFull, inc, m);
        if ((t & 31) >= m) inc += o;
    }
    if ((t & 31) == 31) part[t >> 5] = inc;
    __syncthreads();
    uint32_t run = inc - sum;
    for (int w = 0; w < (t >> 5); ++w) run += part[w];
#pragma unroll
    for (int j = 0; j < kPer; ++j) {
        base[t * kPer + j] = run;
        run += own[j];
    }
    const uint32_t p0 = blockIdx.x * (uint32_t)(kOrderThreads * ITEMS) + t;
    uint32_t rank[ITEMS];
    uint16_t key[ITEMS];
#pragma unroll
    for (int i = 0; i < ITEMS; ++i) {
        const uint32_t p = p0 + (uint32_t)i * kOrderThreads;
        key[i] = p < positions ? keys[p] : kNoSample;
        rank[i] = key[i] != kNoSample ? atomicAdd(&cnt[key[i]], 1u) : 0u;
    }
    __syncthreads();
    uint32_t at[kPer];  // (the reservations in flight together)
#pragma unroll
    for (int j = 0; j < kPer; ++j) {
        const uint32_t c = cnt[t + j * kOrderThreads];
        at[j] = c ? atomicAdd(&cursor[t + j * kOrderThreads], c) : 0u;
    }
#pragma unroll
    for (int j = 0; j < kPer; ++j) base[t + j * kOrderThreads] += at[j];
    __syncthreads();
#pragma unroll
    for (int i = 0; i < ITEMS; ++i)
        if (key[i] != kNoSample) perm[base[key[i]] + rank[i]] = p0 + (uint32_t)i * kOrderThreads;
}

OrderModel order_model(const ModelDev &m)
{
    OrderModel o;
    o.D = std::max((float)-m.a_cmd, 1e-3f);
    o.g = (float)m.g;
    o.rho_a2 = (float)(0.5 * m.rho * m.area);
    o.hl = (float)m.hl;
    o.beta = (float)m.beta;
    o.phi_f = (float)m.phi_f;
    o.thr = (float)m.ttc_thr;
    o.lat = (float)(m.perc_lat * m.dt);
    o.t_max = (float)(m.n_max * m.dt);
    o.lv0 = m.lead_moving ? (float)m.lead_v0 : 0.0f;
    o.lb = (float)m.lead_decel;
    o.lts = (float)m.lead_ts;
    o.lxs = (float)m.lead_xs;
    o.lumped = m.cap_mode == AEB_CAP_LUMPED;
    o.ttc = m.trigger == AEB_TRIGGER_TTC;
    o.lead = m.lead;
    o.moving = m.lead_moving;
    return o;
}

size_t a256(size_t x) { return (x + 255) & ~size_t(255); }

// Scratch of an ordered launch: the ticket counter, the bins' counts and
// cursors (one clear covers the three), the keys and the order.
struct Layout {
    size_t hist = kCounterBytes, cursor = hist + a256(4 * kBins),
           keys = cursor + a256(4 * kBins), perm, bytes;
    explicit Layout(uint64_t positions)
    {
        perm = keys + a256(2 * positions);
        bytes = perm + a256(4 * positions);
    }
};

// Whether a launch of this many positions is worth ordering.
//
// Binary64: a warp gains from lanes of one cap class at any size above one warp
// (its steps take microseconds).
//
// Binary32: the two kernels and the clear cost ~13 us and 24 ns per 1,000
// samples, and rows taken out of order cost more memory traffic; both have to come
// back from steps.  Measured, ordered against index order, over 2e4 .. 1e7 samples
// and horizons of 200 .. 10,000 steps (steps of 1 ms cut short, and whole 10 s
// horizons of coarser steps):
//   - at most one warp per sub-partition (152 x 4 x 32 = 19,456 rollouts) lasts as
//     long as its longest rollout in any order;
//   - below 1,000 steps: 1e6 samples of 200 steps 280 -> 314 us, of 500 572 -> 574,
//     of 700 742 -> 712, of 1,000 995 -> 938; 1e7 of 700 coarse steps 4,021 -> 4,314,
//     of 1,000 4,892 -> 4,818;
//   - samples times steps: 1e8 and more pay (2e4 of 3,000 steps 150 -> 153 us, of
//     5,000 219 -> 210; 4e4 of 2,000 134 -> 135, of 3,000 180 -> 172; 6e4 of 1,000
//     coarse 66 -> 69, of 1,500 83 -> 81; 1e5 of 700 113 -> 115, of 1,000 142 -> 139);
//   - without a lead, a horizon of a few seconds ends every rollout at the same
//     step and only the cap classes gain: 4e8 and 1,500 steps (1e5 of 3,000 steps
//     284 -> 293 us, 2e5 of 2,000 340 -> 340, 4e5 of 1,500 477 -> 477, 1e6 of 1,000
//     829 -> 836, of 1,500 1,176 -> 1,148; at 5 s 1e5 462 -> 450);
//   - the TTC trigger reads two columns more per sample, which counts once the
//     columns no longer stay in the L2: 5e5 and more samples take 2,000 steps (1e6
//     of 1,000 coarse steps 1.05 of index order, of 1,500 0.96, of 2,000 0.89), 2e6
//     and more 3,000 (1e7 of 2,000 1.03; 3e6 of 3,000 0.89);
//   - per-step readings take time that the order does not save: 2e8 and 2,000 steps
//     (4e4 of 3,000 coarse steps 1.01, of 5,000 0.99; 1e5 of 1,500 1.00, of 2,000 0.98).
constexpr uint64_t kTtcMid = uint64_t(1) << 19, kTtcMany = uint64_t(1) << 21;
bool wants_order(uint64_t positions, aeb_precision precision, const ModelDev &m)
{
    if (m.n_max <= 0) return false;
    if (precision == AEB_FP64_PLAIN) return positions > 32;
    if (positions <= 19456) return false;
    const bool ttc = m.trigger == AEB_TRIGGER_TTC, readings = ttc && m.perc;
    const bool cut = !m.lead && m.n_max * m.dt < 4.0;
    const int32_t steps = ttc && positions > kTtcMany               ? 3000
                          : readings || (ttc && positions > kTtcMid) ? 2000
                          : cut                                      ? 1500
                                                                     : 1000;
    const double work = cut ? 4e8 : readings ? 2e8 : 1e8;
    return m.n_max >= steps && (double)positions * m.n_max >= work;
}

size_t order_bytes(uint64_t positions) { return Layout(std::min(positions, kOrderMax)).bytes; }

}  // namespace

size_t rollout_scratch_bytes(uint64_t positions, aeb_precision precision, const ModelDev &m)
{
    return wants_order(positions, precision, m) ? order_bytes(positions) : kCounterBytes;
}

size_t rollout_scratch_bytes_up_to(uint64_t positions, aeb_precision precision, const ModelDev &m)
{
    // (the rule asks for more steps above kTtcMid and kTtcMany, otherwise for fewer)
    for (const uint64_t most : {positions, kTtcMany, kTtcMid})
        if (most <= positions && wants_order(most, precision, m)) return order_bytes(most);
    return kCounterBytes;
}

cudaError_t launch_rollout(const ModelDev &m, const ParamsDev &p, aeb_precision precision,
                           const OutDev &o, const WorkDev &w, const TileDesc *host_tiles,
                           const LaunchCfg &cfg, void *scratch, size_t scratch_bytes,
                           cudaStream_t s)
{
    const uint64_t all = w.tiles ? w.n_tiles * w.tile : w.n;
    const bool order = wants_order(all, precision, m) && scratch_bytes >= order_bytes(all);
    const uint64_t piece = order ? kOrderMax : kNaturalMax;  // positions per launch
    const uint64_t unit = w.tiles ? piece / w.tile : piece;   // tiles or rows per launch
    const uint64_t total = w.tiles ? w.n_tiles : w.n;
    char *base = static_cast<char *>(scratch);
    const Layout lay(std::min(all, kOrderMax));
    for (uint64_t first = 0; first < total; first += unit) {
        const uint64_t len = std::min(unit, total - first);
        WorkDev k = w;
        k.counter = reinterpret_cast<unsigned long long *>(base);
        k.perm = nullptr;
        uint64_t positions = len;
        if (w.tiles) {
            k.tiles = w.tiles + first;
            k.n_tiles = len;
            positions = len * w.tile;
            if (len < total) {
                k.n = 0;
                for (uint64_t t = first; t < first + len; ++t) k.n += host_tiles[t].count;
            }
        } else {
            k.row0 = w.row0 + first;
            k.n = len;
        }
        cudaError_t e = cudaMemsetAsync(base, 0, order ? lay.keys : 2 * sizeof(unsigned long long), s);
        if (e != cudaSuccess) return e;
        if (order) {
            auto *hist = reinterpret_cast<uint32_t *>(base + lay.hist);
            auto *cursor = reinterpret_cast<uint32_t *>(base + lay.cursor);
            auto *keys = reinterpret_cast<uint16_t *>(base + lay.keys);
            auto *perm = reinterpret_cast<uint32_t *>(base + lay.perm);
            const uint32_t np = (uint32_t)positions;
            const uint32_t kb = std::min<uint32_t>((np + kOrderThreads - 1) / kOrderThreads, 152 * 8);
            k_order_keys<<<kb, kOrderThreads, 0, s>>>(order_model(m), p, k, np, hist, keys);
            e = cudaGetLastError();
            if (e != cudaSuccess) return e;
            const bool few = np <= kScatterSmall;
            const uint32_t chunk = (uint32_t)kOrderThreads * (few ? kScatterFew : kScatterMany);
            (few ? k_order_scatter<kScatterFew> : k_order_scatter<kScatterMany>)<<<
                (np + chunk - 1) / chunk, kOrderThreads, 0, s>>>(np, hist, cursor, keys, perm);
            e = cudaGetLastError();
            if (e != cudaSuccess) return e;
            k.perm = perm;
        }
        e = precision == AEB_FP64_PLAIN ? launch_rollout_fp64(m, p, o, k, cfg, s)
                                        : launch_rollout_fp32(m, p, o, k, cfg, s);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

}  // namespace aeb
