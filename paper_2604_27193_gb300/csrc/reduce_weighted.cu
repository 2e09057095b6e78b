// reduce_weighted.cu -- weighted event sums of a set of rollout outputs for
// importance sampling (extension: rare-event estimation of low collision
// probabilities).  Each sample carries the likelihood ratio w of its parameter
// set (nominal over proposal density); the event E of a valid sample is a
// contact, or a final position x_ref beyond x_thr (Sec. VI-C: D_stop > H0).
// The sums Σ w, Σ w², Σ w 1[E], Σ w² 1[E] give the unbiased estimate
// Σ w 1[E] / n of the nominal probability of E and its standard error.
//
// One launch on the caller's stream (after a clear of the sums), in a fixed
// order so that the sums are the same bits for the same inputs: G blocks; block b
// owns samples [b*chunk, (b+1)*chunk); a warp walks its strided share in index
// order and queues the weights of events and of the other valid samples in shared
// memory; 32 queued weights of a kind are then added together (the binary64 unit
// is held 64 cycles or more by a warp instruction whatever its busy lanes, so each weight
// enters one pair of sums, not two; all = events + others).  The block adds its
// threads with a fixed tree and writes one partial; the block that arrives last
// adds the G partials with the same tree.  One pass over 17 bytes per sample
// (status, x_ref, weight).
#include "aeb_internal.h"

namespace aeb {
namespace {

constexpr int kWThreads = 512;
constexpr int kWWarps = kWThreads / 32;
constexpr int kWUnroll = 4;

struct WPart {
    unsigned long long n_valid, n_event;
    double sum_w, sumsq_w, sum_we, sumsq_we;  // w: the samples that are not events
};

__device__ __forceinline__ void wadd(WPart &a, const WPart &b)
{
    a.n_valid += b.n_valid;
    a.n_event += b.n_event;
    a.sum_w += b.sum_w;
    a.sumsq_w += b.sumsq_w;
    a.sum_we += b.sum_we;
    a.sumsq_we += b.sumsq_we;
}

// Fixed-order tree over the block's threads (kWThreads a power of two).
__device__ __forceinline__ void block_tree(WPart &mine, WPart *sh)
{
    const int t = threadIdx.x;
    sh[t] = mine;
    __syncthreads();
    for (int stride = kWThreads / 2; stride > 0; stride >>= 1) {
        if (t < stride) wadd(sh[t], sh[t + stride]);
        __syncthreads();
    }
    mine = sh[0];
    __syncthreads();
}

// x > t for a t that is not NaN (false for a NaN x), on the integer pipe.
__device__ __forceinline__ long long order_key(double x)
{
    const long long b = __double_as_longlong(x);
    return b < 0 ? -(b & 0x7fffffffffffffffll) : b;
}
__device__ __forceinline__ bool above(double x, long long tkey)
{
    const long long mag = __double_as_longlong(x) & 0x7fffffffffffffffll;
    return mag <= 0x7ff0000000000000ll && order_key(x) > tkey;
}

// Queue x of the lanes in `mask`; once 32 weights wait, the warp adds them.
__device__ __forceinline__ void push(double *q, int &fill, unsigned mask, double x, double &sum,
                                     double &sumsq, double one)
{
    const int lane = threadIdx.x & 31;
    if ((mask >> lane) & 1u) q[fill + __popc(mask & ((1u << lane) - 1u))] = x;
    fill += __popc(mask);
    if (fill >= 32) {
        __syncwarp();
        const double y = q[lane], z = q[32 + lane];
        __syncwarp();
        fill -= 32;
        if (lane < fill) q[lane] = z;
        sum = __fma_rn(y, one, sum);
        sumsq = __fma_rn(y, y, sumsq);
        __syncwarp();
    }
}

__global__ void __launch_bounds__(kWThreads, 2)
k_reduce_weighted(const uint8_t *__restrict__ status, const double *__restrict__ x_ref,
                  const double *__restrict__ w, uint64_t n, uint64_t chunk, double x_thr,
                  WPart *parts, aeb_wstats *out)
{
    __shared__ WPart sh[kWThreads];
    __shared__ double q[2][kWWarps][64];
    __shared__ double ones[32];
    __shared__ int last;
    if (threadIdx.x < 32) ones[threadIdx.x] = 1.0;
    __syncthreads();
    const int lane = threadIdx.x & 31, wi = threadIdx.x >> 5;
    const double one = ones[lane];
    const long long tkey = order_key(x_thr);
    WPart a{0ull, 0ull, 0.0, 0.0, 0.0, 0.0};
    int fill_e = 0, fill_o = 0;
    unsigned valid = 0, events = 0;
    const uint64_t lo = (uint64_t)blockIdx.x * chunk;
    const uint64_t hi = (lo + chunk < n) ? lo + chunk : n;
    for (uint64_t base = lo + (uint64_t)wi * 32; base < hi; base += kWThreads * kWUnroll) {
        int s[kWUnroll];
        double x[kWUnroll], v[kWUnroll];
#pragma unroll
        for (int u = 0; u < kWUnroll; ++u) {
            const uint64_t i = base + (uint64_t)u * kWThreads + lane;
            s[u] = AEB_INVALID;
            x[u] = v[u] = 0.0;
            if (i < hi) {
                s[u] = status[i];
                x[u] = x_ref[i];
                v[u] = w[i];
            }
        }
#pragma unroll
        for (int u = 0; u < kWUnroll; ++u) {
            const bool in = s[u] != AEB_INVALID;
            const bool e = in && (s[u] == AEB_CONTACT || above(x[u], tkey));
            const unsigned vm = __ballot_sync(0xffffffffu, in), em = __ballot_sync(0xffffffffu, e);
            valid += __popc(vm);
            events += __popc(em);
            push(q[0][wi], fill_e, em, v[u], a.sum_we, a.sumsq_we, one);
            push(q[1][wi], fill_o, vm & ~em, v[u], a.sum_w, a.sumsq_w, one);
        }
    }
    __syncwarp();
    if (lane < fill_e) {
        const double y = q[0][wi][lane];
        a.sum_we = __fma_rn(y, one, a.sum_we);
        a.sumsq_we = __fma_rn(y, y, a.sumsq_we);
    }
    if (lane < fill_o) {
        const double y = q[1][wi][lane];
        a.sum_w = __fma_rn(y, one, a.sum_w);
        a.sumsq_w = __fma_rn(y, y, a.sumsq_w);
    }
    if (lane == 0) {
        a.n_valid = valid;
        a.n_event = events;
    }
    block_tree(a, sh);
    if (threadIdx.x == 0) {
        parts[blockIdx.x] = a;
        __threadfence();  // the partial is visible before the block counts as arrived
        last = atomicAdd(reinterpret_cast<unsigned long long *>(&out->n), 1ull) ==
               (unsigned long long)gridDim.x - 1ull;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    a = WPart{0ull, 0ull, 0.0, 0.0, 0.0, 0.0};
    for (unsigned b = threadIdx.x; b < gridDim.x; b += kWThreads) {
        const volatile WPart &p = parts[b];  // other blocks' writes
        wadd(a, WPart{p.n_valid, p.n_event, p.sum_w, p.sumsq_w, p.sum_we, p.sumsq_we});
    }
    block_tree(a, sh);
    if (threadIdx.x == 0) {
        out->n = n;
        out->n_valid = a.n_valid;
        out->n_event = a.n_event;
        out->sum_w = a.sum_w + a.sum_we;
        out->sumsq_w = a.sumsq_w + a.sumsq_we;
        out->sum_we = a.sum_we;
        out->sumsq_we = a.sumsq_we;
    }
}

}  // namespace

size_t weighted_partial_bytes() { return sizeof(WPart) * kWMaxBlocks; }

cudaError_t launch_reduce_weighted(const uint8_t *status, const double *x_ref, const double *w,
                                   uint64_t n, double x_thr, void *partials, aeb_wstats *stats,
                                   cudaStream_t s)
{
    // G and chunk depend only on n: blocks of >= 2,048 samples, two per SM at most
    uint64_t g = (n + 2047) / 2048;
    if (g > 304) g = 304;
    if (g < 1) g = 1;
    static_assert(304 <= kWMaxBlocks, "partials");
    const uint64_t chunk = (n + g - 1) / g;
    cudaError_t e = cudaMemsetAsync(stats, 0, sizeof(aeb_wstats), s);
    if (e != cudaSuccess) return e;
    k_reduce_weighted<<<(unsigned)g, kWThreads, 0, s>>>(status, x_ref, w, n, chunk > 0 ? chunk : 1,
                                                        x_thr, static_cast<WPart *>(partials), stats);
    return cudaGetLastError();
}

}  // namespace aeb
