// reduce.cu -- counts, moments, extremes and fixed-bin histograms of a set of
// rollout outputs (Sec. VI-B statistics; Sec. VI-C reads P(D_stop > H0) and the
// safe headways off the stopping-distance histogram).
//
// One launch on the caller's stream (after a clear of the statistics):
//   G blocks; block b owns samples [b*chunk, (b+1)*chunk).  A warp walks its
//   strided share in index order and queues the values that enter a sum (D_stop
//   of a stop, the impact speed of a contact) by kind in shared memory; 32
//   queued values of a kind are then summed, compared and binned together, so
//   the binary64 unit, which a warp instruction holds 64 cycles or more whatever its
//   busy lanes, is paid once per 32 values instead of once per kind and 32
//   samples.  The block combines its lanes in a fixed order into one partial.
//   Histogram bins are counted with shared-memory atomics and flushed with 64-bit global
//   atomics (integer adds commute, so they are exact and order-free).  The
//   block that arrives last adds the G partials in the same fixed pattern.
// G and chunk depend only on n, and so do the queues' contents, so the
// floating-point sums are the same bits on every call.  The work is a single
// pass over 21 bytes per sample (status, x_ref, v_imp, n_steps); bin index and
// extremes are taken from the bits with integer instructions.
#include <cfloat>
#include <cmath>

#include "aeb_internal.h"

namespace aeb {
namespace {

constexpr int kRedThreads = 512;
constexpr int kRedWarps = kRedThreads / 32;
constexpr int kRedUnroll = 2;    // samples a lane loads at a time (4: 1e7 102 against 98 us)

// floor((x - lo) / w) clamped to [0, NBINS - 1] for the power-of-two width
// w = 2^-k.  y = x - lo is one binary64 subtraction, as in the definition; the
// exact scaling by 2^k and the floor are done on its bits with integer
// instructions, which keeps the binary64 pipe (1/64 rate on GB300) for the
// sums.  y = m 2^ex with the 53-bit significand m, so floor(y 2^k) is m shifted
// right by -(ex + k); a normal y with ex + k >= -40 is already >= 2^12.
__device__ __forceinline__ int bin_index(double y, int k)
{
    const long long b = __double_as_longlong(y);
    if (b <= 0) return 0;  // +0, or negative (sign bit set)
    const int e = (int)((b >> 52) & 0x7ff);
    unsigned long long m = (unsigned long long)b & 0xfffffffffffffull;
    int ex = -1074;        // subnormal: y = m 2^-1074
    if (e != 0) {
        m |= 1ull << 52;
        ex = e - 1075;
    }
    const int sh = ex + k;
    if (sh >= -40) return AEB_NBINS - 1;
    const int r = -sh;
    const unsigned long long q = (r >= 64) ? 0ull : (m >> r);
    return q > (unsigned long long)(AEB_NBINS - 1) ? AEB_NBINS - 1 : (int)q;
}

// Total-order key of a double (an involution): the bits for a non-negative
// value, the magnitude bits flipped for a negative one, so that keys compare as
// signed integers in the order of the values (-0 just below +0).  The thread
// loop keeps its extremes as keys, on the integer pipe.
__device__ __forceinline__ long long order_key(long long b)
{
    return b ^ ((b >> 63) & 0x7fffffffffffffffll);
}

// A partial is thirteen 64-bit words of four kinds (RedPartial's order: five
// integer sums, then sum, sum of squares, minimum and maximum of D_stop and of
// the impact speed).  Partials are combined word by word, one warp per word, so
// that the few binary64 additions of a combination run side by side on all
// sub-partitions (13 words in turn took a block ~20 us at any n).
constexpr int kWords = sizeof(RedPartial) / 8;
constexpr int kFinalThreads = 32 * kWords;
static_assert(kWords == 13 && sizeof(RedPartial) == 104, "the words' order below");
enum { kIntSum, kSum, kMin, kMax };
__device__ __forceinline__ int kind_of(int word)
{
    return word < 5 ? kIntSum : (word - 5) % 4 < 2 ? kSum : (word - 5) % 4 == 2 ? kMin : kMax;
}
__device__ __forceinline__ long long identity_of(int kind)
{
    return kind == kMin ? 0x7ff0000000000000ll : kind == kMax ? (long long)0xfff0000000000000ll : 0;
}
// a op b (warp-uniform kind)
__device__ __forceinline__ long long combine(int kind, long long a, long long b)
{
    if (kind == kIntSum) return a + b;
    if (kind == kSum)
        return __double_as_longlong(__longlong_as_double(a) + __longlong_as_double(b));
    const bool less = order_key(b) < order_key(a);
    return less == (kind == kMin) ? b : a;
}
// The warp's lanes' values combined in a fixed order (lane 0 has the result).
__device__ __forceinline__ long long warp_combine(int kind, long long a)
{
#pragma unroll 1
    for (int m = 16; m > 0; m >>= 1) a = combine(kind, a, __shfl_down_sync(0xffffffffu, a, m));
    return a;
}
// Word `word` of the partials [b0, b1), by one warp, in a fixed order.
__device__ __forceinline__ long long combine_partials(const RedPartial *part, uint32_t b0,
                                                      uint32_t b1, int word)
{
    const int kind = kind_of(word);
    long long a = identity_of(kind);
    for (uint32_t j = b0 + (threadIdx.x & 31); j < b1; j += 32)
        a = combine(kind, a, __ldcg(reinterpret_cast<const long long *>(part + j) + word));
    return warp_combine(kind, a);
}

// A lane's running sums of one kind of value, and the warp's queue of values
// still to be added (fewer than 32 between rounds).
struct Moments {
    double sum, sumsq;
    long long kmin, kmax;
};
struct Queue {
    double v[32 + 32];
};

__device__ __forceinline__ void add_value(Moments &m, double x, double one)
{
    m.sum = __fma_rn(x, one, m.sum);  // three register operands: see Queue's use
    m.sumsq = __fma_rn(x, x, m.sumsq);
    const long long b = __double_as_longlong(x), k = order_key(b);
    if ((b & 0x7fffffffffffffffll) > 0x7ff0000000000000ll) return;  // a NaN is no extreme
    m.kmin = k < m.kmin ? k : m.kmin;
    m.kmax = k > m.kmax ? k : m.kmax;
}

// Queue x of the lanes in `mask` (fill: values waiting); once 32 wait, the warp
// adds and bins them.
template <bool HIST, bool SHIFT>
__device__ __forceinline__ void push(Queue &q, int &fill, unsigned mask, double x, Moments &m,
                                     double one, unsigned *hist, double lo, int k)
{
    const int lane = threadIdx.x & 31;
    if ((mask >> lane) & 1u) q.v[fill + __popc(mask & ((1u << lane) - 1u))] = x;
    fill += __popc(mask);
    if (fill >= 32) {
        __syncwarp();
        const double y = q.v[lane], z = q.v[32 + lane];
        __syncwarp();
        fill -= 32;
        if (lane < fill) q.v[lane] = z;
        add_value(m, y, one);
        if (HIST) atomicAdd(&hist[bin_index(SHIFT ? __fma_rn(lo, -one, y) : y, k)], 1u);
        __syncwarp();
    }
}
template <bool HIST, bool SHIFT>
__device__ __forceinline__ void drain(const Queue &q, int fill, Moments &m, double one,
                                      unsigned *hist, double lo, int k)
{
    __syncwarp();
    const int lane = threadIdx.x & 31;
    if (lane < fill) {
        const double y = q.v[lane];
        add_value(m, y, one);
        if (HIST) atomicAdd(&hist[bin_index(SHIFT ? __fma_rn(lo, -one, y) : y, k)], 1u);
    }
}

template <class Out>
__device__ __forceinline__ void store_partial(Out *out, const RedPartial &acc, uint64_t n)
{
    out->n = n;
    out->n_stop = acc.n_stop;
    out->n_contact = acc.n_contact;
    out->n_horizon = acc.n_horizon;
    out->n_invalid = acc.n_invalid;
    out->steps = acc.steps;
    out->sum_d = acc.sum_d;
    out->sumsq_d = acc.sumsq_d;
    out->min_d = acc.min_d;
    out->max_d = acc.max_d;
    out->sum_v = acc.sum_v;
    out->sumsq_v = acc.sumsq_v;
    out->min_v = acc.min_v;
    out->max_v = acc.max_v;
}

// With histograms, followed by 2 AEB_NBINS counters.
struct RedShared {
    union {
        struct {
            Queue d[kRedWarps], v[kRedWarps];
        } q;
        long long word[kWords - 4][kRedThreads];  // the lanes' words from the fifth on
    };
    unsigned count[4][kRedWarps];  // the warps' first four
    RedPartial part;
    double one[32];
    int last;
};
static_assert(sizeof(RedShared) + 8 * AEB_NBINS <= 96 * 1024, "two blocks per SM");

// SHIFT: an origin of the histograms is not 0 (without one the subtraction is
// left out: x - 0 is x; 1e7 samples 98 -> 78 us).
// What bounds it: the binary64 unit, 76 % busy.  Counted without SHIFT: three warp
// instructions of that unit per 32 values, one more than the two written, each
// holding it 73 cycles (k_reduce_weighted: the two written, 77 cycles); the
// rollout kernel's register forms take 65.
// HIST: accumulate the two histograms and let the last block finish the
// statistics (the count in stats->n, clear at launch, tells which one that is).
// With a block table, block b reduces rows [out_offset + first, + count) of job
// table[b].job (a segment of one job), otherwise rows [b chunk, (b+1) chunk) of
// [0, n).
template <bool HIST, bool SHIFT>
__global__ void __launch_bounds__(kRedThreads, 2)
k_reduce_partial(const uint8_t *__restrict__ st, const double *__restrict__ xr,
                 const double *__restrict__ vi, const int32_t *__restrict__ ns, uint64_t n,
                 uint64_t chunk, const TileDesc *__restrict__ table, const JobDev *__restrict__ jobs,
                 aeb_hist_spec h, int k_d, int k_v, RedPartial *__restrict__ part,
                 aeb_stats *__restrict__ stats)
{
    extern __shared__ char smem[];
    RedShared &sh = *reinterpret_cast<RedShared *>(smem);
    unsigned *sh_d = reinterpret_cast<unsigned *>(smem + sizeof(RedShared));
    unsigned *sh_v = sh_d + AEB_NBINS;
    if (threadIdx.x < 32) sh.one[threadIdx.x] = 1.0;
    if (HIST)
        for (int j = threadIdx.x; j < 2 * AEB_NBINS; j += kRedThreads) sh_d[j] = 0u;
    __syncthreads();

    uint64_t lo, hi;
    if (table) {
        const TileDesc d = table[blockIdx.x];
        lo = jobs[d.job].out_offset + d.first;
        hi = lo + d.count;
    } else {
        lo = (uint64_t)blockIdx.x * chunk;
        hi = (lo + chunk < n) ? lo + chunk : n;
    }
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const double one = sh.one[lane];  // a register the compiler cannot take for a constant
    Moments md{0.0, 0.0, order_key(0x7ff0000000000000ll), order_key(0xfff0000000000000ll)}, mv = md;
    int fill_d = 0, fill_v = 0;
    unsigned long long steps = 0;
    unsigned n_stop = 0, n_contact = 0, n_horizon = 0, n_invalid = 0;  // of the warp
    for (uint64_t base = lo + (uint64_t)w * 32; base < hi; base += kRedThreads * kRedUnroll) {
        // the loads of kRedUnroll rounds first: a block a SM or two must keep
        // the memory busy
        int s[kRedUnroll], c[kRedUnroll];
        double x[kRedUnroll], v[kRedUnroll];
#pragma unroll
        for (int u = 0; u < kRedUnroll; ++u) {
            const uint64_t i = base + (uint64_t)u * kRedThreads + lane;
            s[u] = -1;
            c[u] = 0;
            x[u] = v[u] = 0.0;
            if (i < hi) {
                s[u] = st[i];
                c[u] = ns[i];
                x[u] = xr[i];
                v[u] = vi[i];
            }
        }
#pragma unroll
        for (int u = 0; u < kRedUnroll; ++u) {
            const unsigned in = __ballot_sync(0xffffffffu, s[u] >= 0);
            const unsigned stop = __ballot_sync(0xffffffffu, s[u] == AEB_STOP);
            const unsigned contact = __ballot_sync(0xffffffffu, s[u] == AEB_CONTACT);
            const unsigned horizon = __ballot_sync(0xffffffffu, s[u] == AEB_HORIZON);
            n_stop += __popc(stop);
            n_contact += __popc(contact);
            n_horizon += __popc(horizon);
            n_invalid += __popc(in & ~(stop | contact | horizon));
            steps += (unsigned long long)(long long)c[u];
            push<HIST, SHIFT>(sh.q.d[w], fill_d, stop, x[u], md, one, sh_d, h.lo_d, k_d);
            push<HIST, SHIFT>(sh.q.v[w], fill_v, contact, v[u], mv, one, sh_v, h.lo_v, k_v);
        }
    }
    drain<HIST, SHIFT>(sh.q.d[w], fill_d, md, one, sh_d, h.lo_d, k_d);
    drain<HIST, SHIFT>(sh.q.v[w], fill_v, mv, one, sh_v, h.lo_v, k_v);
    __syncthreads();  // the queues' memory is used anew
    const long long word[kWords - 4] = {
        (long long)steps, __double_as_longlong(md.sum), __double_as_longlong(md.sumsq),
        order_key(md.kmin), order_key(md.kmax), __double_as_longlong(mv.sum),
        __double_as_longlong(mv.sumsq), order_key(mv.kmin), order_key(mv.kmax)};
#pragma unroll
    for (int j = 0; j < kWords - 4; ++j) sh.word[j][threadIdx.x] = word[j];
    if (lane == 0) {
        sh.count[0][w] = n_stop;
        sh.count[1][w] = n_contact;
        sh.count[2][w] = n_horizon;
        sh.count[3][w] = n_invalid;
    }
    __syncthreads();
    if (w < kWords) {
        const int kind = kind_of(w);
        long long a = identity_of(kind);
        if (w < 4) {
            if (lane < kRedWarps) a = sh.count[w][lane];
        } else {
            a = sh.word[w - 4][lane];
            for (int j = 1; j < kRedWarps; ++j) a = combine(kind, a, sh.word[w - 4][32 * j + lane]);
        }
        a = warp_combine(kind, a);
        if (lane == 0) reinterpret_cast<long long *>(part + blockIdx.x)[w] = a;
    }
    if (!HIST) return;
    for (int j = threadIdx.x; j < AEB_NBINS; j += kRedThreads) {
        if (sh_d[j]) atomicAdd(reinterpret_cast<unsigned long long *>(&stats->hist_d[j]),
                               (unsigned long long)sh_d[j]);
        if (sh_v[j]) atomicAdd(reinterpret_cast<unsigned long long *>(&stats->hist_v[j]),
                               (unsigned long long)sh_v[j]);
    }
    __threadfence();  // the partial is visible before the block counts as arrived
    __syncthreads();
    if (threadIdx.x == 0)
        sh.last = atomicAdd(reinterpret_cast<unsigned long long *>(&stats->n), 1ull) ==
                  (unsigned long long)gridDim.x - 1ull;
    __syncthreads();
    if (!sh.last) return;
    __threadfence();
    if (w < kWords) {
        const long long a = combine_partials(part, 0, gridDim.x, w);
        if (lane == 0) reinterpret_cast<long long *>(&sh.part)[w] = a;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        store_partial(stats, sh.part, n);
        stats->lo_d = h.lo_d;
        stats->w_d = h.w_d;
        stats->lo_v = h.lo_v;
        stats->w_v = h.w_v;
    }
}

// Block j adds the partials [first[j], first[j+1]) of job j in index order.
__global__ void __launch_bounds__(kFinalThreads)
k_reduce_jobs_final(const RedPartial *__restrict__ part, const uint32_t *__restrict__ first,
                    const JobDev *__restrict__ jobs, aeb_job_stats *__restrict__ out)
{
    __shared__ RedPartial sum;
    const int w = threadIdx.x >> 5;
    const long long a = combine_partials(part, first[blockIdx.x], first[blockIdx.x + 1], w);
    if ((threadIdx.x & 31) == 0) reinterpret_cast<long long *>(&sum)[w] = a;
    __syncthreads();
    if (threadIdx.x == 0) store_partial(out + blockIdx.x, sum, jobs[blockIdx.x].n);
}

}  // namespace

// Blocks: one per 2,048 samples (four per thread) up to 256, so that small
// reductions spread over the SMs; beyond 2^21 samples two per SM, each with
// room to stream.
int reduce_blocks_for(uint64_t n)
{
    if (n > (uint64_t(1) << 21)) return 304;
    const uint64_t g = (n + 2047) / 2048;
    return g < 1 ? 1 : g > 256 ? 256 : (int)g;
}

cudaError_t launch_reduce(const uint8_t *status, const double *x_ref, const double *v_imp,
                          const int32_t *n_steps, uint64_t n, const aeb_hist_spec &h,
                          RedPartial *partials, aeb_stats *stats, cudaStream_t s)
{
    const int g = reduce_blocks_for(n);
    const uint64_t chunk = (n + (uint64_t)g - 1) / (uint64_t)g;
    constexpr int kBytes = (int)(sizeof(RedShared) + 2 * sizeof(unsigned) * AEB_NBINS);
    auto kern = (h.lo_d != 0.0 || h.lo_v != 0.0) ? k_reduce_partial<true, true>
                                                 : k_reduce_partial<true, false>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kBytes);
    if (e == cudaSuccess) e = cudaMemsetAsync(stats, 0, sizeof(aeb_stats), s);
    if (e != cudaSuccess) return e;
    kern<<<g, kRedThreads, kBytes, s>>>(status, x_ref, v_imp, n_steps, n, chunk, nullptr, nullptr, h,
                                        -std::ilogb(h.w_d), -std::ilogb(h.w_v), partials, stats);
    return cudaGetLastError();
}

cudaError_t launch_reduce_jobs(const uint8_t *status, const double *x_ref, const double *v_imp,
                               const int32_t *n_steps, const TileDesc *blocks, uint32_t n_blocks,
                               const uint32_t *first, const JobDev *jobs, uint32_t n_jobs,
                               RedPartial *partials, aeb_job_stats *stats, cudaStream_t s)
{
    if (n_blocks > 0) {
        k_reduce_partial<false, false><<<n_blocks, kRedThreads, sizeof(RedShared), s>>>(
            status, x_ref, v_imp, n_steps, 0, 0, blocks, jobs, aeb_hist_spec{}, 0, 0, partials,
            nullptr);
        const cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    k_reduce_jobs_final<<<n_jobs, kFinalThreads, 0, s>>>(partials, first, jobs, stats);
    return cudaGetLastError();
}

}  // namespace aeb
