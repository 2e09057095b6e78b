// rollout_common.cuh -- pieces shared by the FP64 and FP32-compensated rollout
// kernels: the warp work queue (lane refill), the per-sample validity test, the
// step-count rule and the output store.
#pragma once

#include "aeb_internal.h"

namespace aeb {

constexpr unsigned kFull = 0xffffffffu;

__device__ __forceinline__ unsigned lanemask_lt()
{
    unsigned m;
    asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
    return m;
}

// The rows of a position: parameters, outputs, perception key, and the TTC
// threshold of its job.
struct Row {
    uint64_t p, o, k;
    double thr;
};
__device__ __forceinline__ Row row_of(const WorkDev &w, uint32_t pos, double model_thr)
{
    Row r;
    if (!w.tiles) {
        r.p = r.o = w.row0 + pos;
        r.k = w.key_base + r.p;
        r.thr = model_thr;
    } else {
        const uint32_t t = pos / w.tile;
        const TileDesc d = w.tiles[t];
        const JobDev j = w.jobs[d.job];
        const uint64_t i = d.first + (pos - t * w.tile);
        r.p = j.param_offset + i;
        r.o = j.out_offset + i;
        r.k = j.key_offset + i;
        r.thr = j.ttc_thr;
    }
    return r;
}

// A claimed ticket: entries [start, start + count) of the processing order.
// Warp-uniform.
struct Ticket {
    uint32_t start;
    int count;
    bool ok;
};

// Claim the next ticket (all 32 lanes call together; lane 0 takes it).
__device__ __forceinline__ Ticket claim_ticket(const WorkDev &w)
{
    unsigned long long t = 0;
    if ((threadIdx.x & 31u) == 0) t = atomicAdd(w.counter, 1ull);
    t = __shfl_sync(kFull, t, 0);
    Ticket r;
    const uint64_t start = (uint64_t)t * w.tile;
    r.start = (uint32_t)start;
    if (w.tiles && !w.perm) {
        r.ok = t < w.n_tiles;
        r.count = r.ok ? (int)w.tiles[t].count : 0;
    } else {
        r.ok = start < w.n;
        r.count = r.ok ? (int)((w.n - start < (uint64_t)w.tile) ? w.n - start : w.tile) : 0;
    }
    return r;
}
__device__ __forceinline__ uint32_t position(const WorkDev &w, uint32_t entry)
{
    return w.perm ? __ldg(w.perm + entry) : entry;
}

// Number of tickets a launch hands out.
__host__ __forceinline__ uint64_t tickets_of(const WorkDev &w)
{
    return (w.tiles && !w.perm) ? w.n_tiles : (w.n + w.tile - 1) / w.tile;
}

// Philox-4x64-10 (Salmon, Moraes, Dror, Shaw, SC 2011): the block of counter
// c under key (k0, k1), in place.  Used for the per-step perception readings
// of the TTC trigger, two readings per block: counter (parameter row,
// floor(k / 2), 0, 0), key (seed, kPercKey1) (see perc_halves).
constexpr uint64_t kPercKey1 = 0x5045524345505431ull;  // "PERCEPT1"
__device__ __forceinline__ void philox_block(uint64_t c[4], uint64_t k0, uint64_t k1)
{
    constexpr uint64_t kM0 = 0xD2E7470EE14C6C93ull, kM1 = 0xCA5A826395121157ull;
    constexpr uint64_t kW0 = 0x9E3779B97F4A7C15ull, kW1 = 0xBB67AE8584CAA73Bull;
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        const uint64_t h0 = __umul64hi(kM0, c[0]), l0 = kM0 * c[0];
        const uint64_t h1 = __umul64hi(kM1, c[2]), l1 = kM1 * c[2];
        const uint64_t n0 = h1 ^ c[1] ^ k0, n2 = h0 ^ c[3] ^ k1;
        c[0] = n0;
        c[1] = l1;
        c[2] = n2;
        c[3] = l0;
        k0 += kW0;
        k1 += kW1;
    }
}

// The four 32-bit words h_j of reading k (taken at step k) of parameter row
// `row`: the high halves of the block's words for even k, the low halves for
// odd k.  Uniforms u_j = h_j 2^-32; the reading is missing if u_4 is below
// the dropout probability.
__device__ __forceinline__ void perc_halves(uint64_t row, uint64_t k, uint64_t seed, uint32_t h[4])
{
    uint64_t c[4] = {row, k >> 1, 0, 0};
    philox_block(c, seed, kPercKey1);
    const int sh = (k & 1) ? 0 : 32;
#pragma unroll
    for (int j = 0; j < 4; ++j) h[j] = (uint32_t)(c[j] >> sh);
}

// A sample is invalid if any field is not finite, mass <= 0, or tau, mu, C_d
// or the delay is negative.
__device__ __forceinline__ bool sample_valid(const double f[AEB_NFIELDS])
{
#pragma unroll
    for (int j = 0; j < AEB_NFIELDS; ++j)
        if (!isfinite(f[j])) return false;
    if (!(f[kMass] > 0.0) || f[kTau] < 0.0 || f[kMu] < 0.0 || f[kCd] < 0.0 || f[kTdelay] < 0.0)
        return false;
    return true;
}

// Smallest n >= 0 with (double)n * dt >= t (clamped to 2^31 - 1).  The
// adjustment loops make the result independent of how the first guess rounds.
__device__ __forceinline__ int32_t steps_to_reach_dev(double t, double dt)
{
    if (!(t > 0.0)) return 0;
    double q = ceil(t / dt);
    if (!(q <= 2147483647.0)) return 2147483647;
    long long n = (long long)q;
    while (n > 0 && (double)(n - 1) * dt >= t) --n;
    while ((double)n * dt < t) ++n;
    return (int32_t)n;
}

__device__ __forceinline__ void store_out(const OutDev &o, uint64_t i, uint8_t status,
                                          double x_raw, double x_ref, double v_imp,
                                          double t_end, int32_t n_steps, int32_t n_onset)
{
    if (o.status) o.status[i] = status;
    if (o.x_raw) o.x_raw[i] = x_raw;
    if (o.x_ref) o.x_ref[i] = x_ref;
    if (o.v_imp) o.v_imp[i] = v_imp;
    if (o.t_end) o.t_end[i] = t_end;
    if (o.n_steps) o.n_steps[i] = n_steps;
    if (o.n_onset) o.n_onset[i] = n_onset;
}

__device__ __forceinline__ void load_fields(const ParamsDev &p, uint64_t i, double f[AEB_NFIELDS])
{
#pragma unroll
    for (int j = 0; j < AEB_NFIELDS; ++j) f[j] = __ldg(p.col[j] + i);
}

}  // namespace aeb
