// batch.cpp -- batched launches: many jobs (scenarios, thresholds) with uneven
// sample counts in one persistent rollout launch over a (job, tile) work table,
// followed by a per-job fixed-order reduction, captured once as a CUDA graph.
// Also the launch-shape configuration and its autotuner.
#include <cmath>
#include <cstdio>
#include <cstring>
#include <fstream>
#include <sstream>
#include <string>
#include <vector>

#include "aeb_internal.h"
#include "host_util.h"

struct aeb_batch {
    int device = 0;
    uint32_t n_jobs = 0;
    void *mem = nullptr;
    cudaGraph_t graph = nullptr;
    cudaGraphExec_t exec = nullptr;
};

namespace aeb {
namespace {

size_t a256(size_t x) { return (x + 255) & ~size_t(255); }

bool valid_precision(aeb_precision p) { return p == AEB_FP64_PLAIN || p == AEB_FP32_COMP; }

aeb_status check_cfg(aeb_precision precision, const aeb_launch_config &c)
{
    if (!valid_precision(precision)) return fail(AEB_EINVAL, "unknown precision");
    if (c.tile < 32 || c.tile > 256 || c.tile % 32)
        return fail(AEB_EINVAL, "launch config: tile must be a multiple of 32 in [32, 256]");
    if (c.blocks_per_sm < 0 || c.blocks_per_sm > 32)
        return fail(AEB_EINVAL, "launch config: blocks_per_sm must be in [0, 32]");
    return AEB_OK;
}

void destroy_plan(aeb_batch *b)
{
    if (!b) return;
    if (b->exec) cudaGraphExecDestroy(b->exec);
    if (b->graph) cudaGraphDestroy(b->graph);
    if (b->mem) cudaFree(b->mem);  // waits for work still using it
    delete b;
}

// A batched call, checked and laid out: its tables on the host, in one block as
// they go to the device (jobs, tiles, reduction segments, each job's first
// segment), then the partials and the rollout's scratch.
struct Layout {
    ModelDev md;
    ParamsDev pd;
    LaunchCfg cfg;
    uint32_t T = 0;
    uint64_t total = 0;  // samples
    std::vector<JobDev> jobs;
    std::vector<TileDesc> tiles, red;
    std::vector<uint32_t> first;
    size_t o_tiles = 0, o_red = 0, o_first = 0, o_part = 0, o_scratch = 0;
    size_t scratch = 0;  // bytes
    size_t bytes() const { return o_scratch + scratch; }
};

aeb_status lay_out(const char *who, const aeb_model *model, const aeb_job *jobs, uint32_t n_jobs,
                   const aeb_params *params, aeb_precision precision, const aeb_outputs *out,
                   const aeb_job_stats *stats, Layout *L)
{
    const std::string w = who;
    if (!jobs || n_jobs == 0 || !stats || !out)
        return fail(AEB_EINVAL, w + ": NULL argument or no jobs");
    aeb_status st = check_model(model, &L->md);
    if (st != AEB_OK) return st;
    st = check_params(params, &L->pd);
    if (st != AEB_OK) return st;
    if (!valid_precision(precision)) return fail(AEB_EINVAL, "unknown precision");
    if (!out->status || !out->x_ref || !out->v_imp || !out->n_steps)
        return fail(AEB_EINVAL, w + ": status, x_ref, v_imp and n_steps are required");
    if (reinterpret_cast<uintptr_t>(stats) % 8 != 0)
        return fail(AEB_EINVAL, w + ": stats is not 8-byte aligned");
    L->cfg = launch_cfg(precision);
    const uint32_t T = L->T = (uint32_t)L->cfg.tile;
    L->jobs.resize(n_jobs);
    L->first.resize(n_jobs + 1);
    for (uint32_t j = 0; j < n_jobs; ++j) {
        const aeb_job &jb = jobs[j];
        if (!std::isfinite(jb.ttc_thr)) return fail(AEB_EINVAL, w + ": ttc_thr not finite");
        L->jobs[j] = JobDev{jb.param_offset, jb.out_offset, jb.n, jb.ttc_thr, jb.key_offset};
        for (uint64_t f = 0; f < jb.n; f += T)
            L->tiles.push_back(TileDesc{f, j, (uint32_t)std::min<uint64_t>(T, jb.n - f)});
        L->first[j] = (uint32_t)L->red.size();
        for (uint64_t f = 0; f < jb.n; f += kRedSegment)
            L->red.push_back(TileDesc{f, j, (uint32_t)std::min<uint64_t>(kRedSegment, jb.n - f)});
        if (L->red.size() > 0xffffffffull) return fail(AEB_EINVAL, w + ": too many reduction segments");
        L->total += jb.n;
    }
    L->first[n_jobs] = (uint32_t)L->red.size();
    L->o_tiles = a256(sizeof(JobDev) * n_jobs);
    L->o_red = L->o_tiles + a256(sizeof(TileDesc) * L->tiles.size());
    L->o_first = L->o_red + a256(sizeof(TileDesc) * L->red.size());
    L->o_part = L->o_first + a256(sizeof(uint32_t) * L->first.size());
    L->o_scratch = L->o_part + a256(sizeof(RedPartial) * (L->red.size() + 1));
    L->scratch = rollout_scratch_bytes((uint64_t)L->tiles.size() * T, precision, L->md);
    return AEB_OK;
}

// The tables in one block, as they lie on the device.
std::vector<char> packed(const Layout &L)
{
    std::vector<char> b(L.o_part);
    std::memcpy(b.data(), L.jobs.data(), sizeof(JobDev) * L.jobs.size());
    if (!L.tiles.empty())
        std::memcpy(b.data() + L.o_tiles, L.tiles.data(), sizeof(TileDesc) * L.tiles.size());
    if (!L.red.empty()) std::memcpy(b.data() + L.o_red, L.red.data(), sizeof(TileDesc) * L.red.size());
    std::memcpy(b.data() + L.o_first, L.first.data(), sizeof(uint32_t) * L.first.size());
    return b;
}

// The rollouts and the per-job reduction, with the tables at `base` on the device.
cudaError_t enqueue(const Layout &L, aeb_precision precision, const aeb_outputs *out,
                    aeb_job_stats *stats, char *base, cudaStream_t s)
{
    const auto *jobs = reinterpret_cast<const JobDev *>(base);
    const auto *tiles = reinterpret_cast<const TileDesc *>(base + L.o_tiles);
    const auto *red = reinterpret_cast<const TileDesc *>(base + L.o_red);
    const auto *first = reinterpret_cast<const uint32_t *>(base + L.o_first);
    if (!L.tiles.empty()) {
        const WorkDev w{L.total, L.T, nullptr, tiles, (uint64_t)L.tiles.size(), jobs, 0, 0, nullptr};
        const cudaError_t e = launch_rollout(L.md, L.pd, precision, out_dev(out), w, L.tiles.data(),
                                             L.cfg, base + L.o_scratch, L.scratch, s);
        if (e != cudaSuccess) return e;
    }
    return launch_reduce_jobs(out->status, out->x_ref, out->v_imp, out->n_steps, red,
                              (uint32_t)L.red.size(), first, jobs, (uint32_t)L.jobs.size(),
                              reinterpret_cast<RedPartial *>(base + L.o_part), stats, s);
}

}  // namespace
}  // namespace aeb

using namespace aeb;

extern "C" aeb_status aeb_batch_create(const aeb_model *model, const aeb_job *jobs, uint32_t n_jobs,
                                       const aeb_params *params, aeb_precision precision,
                                       const aeb_outputs *out, aeb_job_stats *stats,
                                       aeb_batch **plan)
{
    clear_error();
    if (!plan) return fail(AEB_EINVAL, "aeb_batch_create: plan is NULL");
    *plan = nullptr;
    Layout L;
    aeb_status st = lay_out("aeb_batch_create", model, jobs, n_jobs, params, precision, out, stats, &L);
    if (st != AEB_OK) return st;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return cuda_fail(e, "cudaGetDevice");

    aeb_batch *b = new aeb_batch;
    b->device = dev;
    b->n_jobs = n_jobs;
    e = cudaMalloc(&b->mem, L.bytes());
    if (e == cudaErrorMemoryAllocation && L.scratch > kCounterBytes) {
        cudaGetLastError();
        L.scratch = kCounterBytes;  // no room for a processing order: natural order
        e = cudaMalloc(&b->mem, L.bytes());
    }
    if (e != cudaSuccess) {
        delete b;
        return cuda_fail(e, "cudaMalloc(batch plan)");
    }
    char *base = static_cast<char *>(b->mem);
    const std::vector<char> tables = packed(L);
    e = cudaMemcpy(base, tables.data(), tables.size(), cudaMemcpyHostToDevice);
    if (e != cudaSuccess) {
        destroy_plan(b);
        return cuda_fail(e, "cudaMemcpy(batch tables)");
    }
    cudaStream_t cs = nullptr;
    e = cudaStreamCreateWithFlags(&cs, cudaStreamNonBlocking);
    if (e != cudaSuccess) {
        destroy_plan(b);
        return cuda_fail(e, "cudaStreamCreate");
    }
    e = cudaStreamBeginCapture(cs, cudaStreamCaptureModeThreadLocal);
    if (e == cudaSuccess) {
        const cudaError_t le = enqueue(L, precision, out, stats, base, cs);
        e = cudaStreamEndCapture(cs, &b->graph);
        if (le != cudaSuccess) e = le;
    }
    if (e == cudaSuccess) e = cudaGraphInstantiate(&b->exec, b->graph, 0);
    cudaStreamDestroy(cs);
    if (e != cudaSuccess) {
        destroy_plan(b);
        return cuda_fail(e, "batch graph capture");
    }
    *plan = b;
    return AEB_OK;
}

extern "C" aeb_status aeb_batch_run(aeb_batch *plan, void *stream)
{
    clear_error();
    if (!plan) return fail(AEB_EINVAL, "aeb_batch_run: plan is NULL");
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return cuda_fail(e, "cudaGetDevice");
    if (dev != plan->device) return fail(AEB_EINVAL, "aeb_batch_run: plan belongs to another device");
    e = cudaGraphLaunch(plan->exec, static_cast<cudaStream_t>(stream));
    if (e != cudaSuccess) return cuda_fail(e, "cudaGraphLaunch");
    return AEB_OK;
}

extern "C" void aeb_batch_destroy(aeb_batch *plan) { destroy_plan(plan); }

extern "C" aeb_status aeb_rollout_batched(const aeb_model *model, const aeb_job *jobs,
                                          uint32_t n_jobs, const aeb_params *params,
                                          aeb_precision precision, const aeb_outputs *out,
                                          aeb_job_stats *stats, void *stream)
{
    // One shot: no graph, and memory from the library's pool where it has some
    // (otherwise as a plan).
    clear_error();
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    Layout L;
    aeb_status st = lay_out("aeb_batch_create", model, jobs, n_jobs, params, precision, out, stats, &L);
    if (st != AEB_OK) return st;
    cudaError_t e = cudaSuccess;
    if (char *base = static_cast<char *>(pool_alloc(L.bytes(), s))) {
        const std::vector<char> tables = packed(L);
        e = cudaMemcpyAsync(base, tables.data(), tables.size(), cudaMemcpyHostToDevice, s);
        if (e == cudaSuccess) e = enqueue(L, precision, out, stats, base, s);
        const cudaError_t f = cudaFreeAsync(base, s), g = cudaStreamSynchronize(s);
        if (e == cudaSuccess) e = f != cudaSuccess ? f : g;
        return e == cudaSuccess ? AEB_OK : cuda_fail(e, "batched rollout");
    }
    aeb_batch *b = nullptr;
    st = aeb_batch_create(model, jobs, n_jobs, params, precision, out, stats, &b);
    if (st != AEB_OK) return st;
    st = aeb_batch_run(b, stream);
    if (st == AEB_OK) {
        e = cudaStreamSynchronize(s);
        if (e != cudaSuccess) st = cuda_fail(e, "cudaStreamSynchronize");
    }
    destroy_plan(b);
    return st;
}

extern "C" aeb_status aeb_get_launch_config(aeb_precision precision, aeb_launch_config *cfg)
{
    clear_error();
    if (!cfg) return fail(AEB_EINVAL, "aeb_get_launch_config: cfg is NULL");
    if (!valid_precision(precision)) return fail(AEB_EINVAL, "unknown precision");
    const LaunchCfg c = launch_cfg(precision);
    cfg->tile = c.tile;
    cfg->blocks_per_sm = c.blocks_per_sm;
    return AEB_OK;
}

extern "C" aeb_status aeb_set_launch_config(aeb_precision precision, const aeb_launch_config *cfg)
{
    clear_error();
    if (!cfg) return fail(AEB_EINVAL, "aeb_set_launch_config: cfg is NULL");
    const aeb_status st = check_cfg(precision, *cfg);
    if (st != AEB_OK) return st;
    LaunchCfg c = launch_cfg(precision);
    c.tile = cfg->tile;
    c.blocks_per_sm = cfg->blocks_per_sm;
    set_launch_cfg(precision, c);
    return AEB_OK;
}

namespace aeb {
namespace {

// Cache lines: "<key> <tile> <blocks_per_sm>", key = device|sms|precision|cap|trigger|lead.
std::string tune_key(const aeb_model &m, aeb_precision precision)
{
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaDeviceProp prop;
    std::string name = "unknown";
    if (cudaGetDeviceProperties(&prop, dev) == cudaSuccess) name = prop.name;
    for (char &c : name)
        if (c == ' ') c = '_';
    std::ostringstream k;
    k << name << "|" << sms << "|" << precision << "|" << m.cap_mode << "|" << m.trigger << "|"
      << m.lead;
    return k.str();
}

bool cache_lookup(const char *path, const std::string &key, aeb_launch_config *out)
{
    std::ifstream f(path);
    std::string k;
    int t, b;
    while (f >> k >> t >> b)
        if (k == key) {
            out->tile = t;
            out->blocks_per_sm = b;
            return true;
        }
    return false;
}

void cache_store(const char *path, const std::string &key, const aeb_launch_config &c)
{
    std::vector<std::string> lines;
    {
        std::ifstream f(path);
        std::string line;
        while (std::getline(f, line))
            if (line.compare(0, key.size() + 1, key + " ") != 0 && !line.empty()) lines.push_back(line);
    }
    std::ofstream f(path, std::ios::trunc);
    for (const auto &l : lines) f << l << "\n";
    f << key << " " << c.tile << " " << c.blocks_per_sm << "\n";
}

}  // namespace
}  // namespace aeb

extern "C" aeb_status aeb_autotune(const aeb_model *model, const aeb_params *params, uint64_t n,
                                   aeb_precision precision, const aeb_outputs *out, void *stream,
                                   const char *cache_path, aeb_launch_config *best)
{
    clear_error();
    if (!best || !out || n == 0) return fail(AEB_EINVAL, "aeb_autotune: NULL argument or n == 0");
    if (!valid_precision(precision)) return fail(AEB_EINVAL, "unknown precision");
    ModelDev md;
    aeb_status st = check_model(model, &md);
    if (st != AEB_OK) return st;
    const std::string key = tune_key(*model, precision);
    if (cache_path && cache_lookup(cache_path, key, best) && check_cfg(precision, *best) == AEB_OK)
        return aeb_set_launch_config(precision, best);

    cudaStream_t s = static_cast<cudaStream_t>(stream);
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    if (cudaEventCreate(&e0) != cudaSuccess || cudaEventCreate(&e1) != cudaSuccess)
        return fail(AEB_ECUDA, "aeb_autotune: cudaEventCreate failed");
    const LaunchCfg saved = launch_cfg(precision);
    const int tl[] = {32, 64, 128};
    float best_ms = 1e30f;
    aeb_launch_config win{saved.tile, saved.blocks_per_sm};
    for (int ti = 0; ti < 3 && st == AEB_OK; ++ti) {
        for (int bps = 3; bps <= 8 && st == AEB_OK; ++bps) {
            LaunchCfg c = saved;
            c.tile = tl[ti];
            c.blocks_per_sm = bps;
            set_launch_cfg(precision, c);
            float ms = 0.0f;
            for (int rep = 0; rep < 2 && st == AEB_OK; ++rep) {  // warm-up, then timed
                cudaEventRecord(e0, s);
                st = aeb_rollout(model, params, n, precision, out, stream);
                cudaEventRecord(e1, s);
                if (cudaEventSynchronize(e1) != cudaSuccess) st = fail(AEB_ECUDA, "aeb_autotune: sync");
                cudaEventElapsedTime(&ms, e0, e1);
            }
            if (st == AEB_OK && ms < best_ms) {
                best_ms = ms;
                win = aeb_launch_config{c.tile, c.blocks_per_sm};
            }
        }
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    set_launch_cfg(precision, saved);
    if (st != AEB_OK) return st;
    *best = win;
    if (cache_path) cache_store(cache_path, key, win);
    return aeb_set_launch_config(precision, &win);
}
