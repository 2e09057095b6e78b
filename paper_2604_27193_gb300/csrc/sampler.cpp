// sampler.cpp -- deterministic host sampling of parameter sets (Sec. IV-A,
// IV-C: random numbers are drawn on the CPU from a fixed seed and the
// parameter vectors are then transferred to the GPU).
//
// Counter-based: sample i, quantity q draws from Philox-4x64-10 (Salmon et al.,
// SC'11) at counter (i, q / 2, 0, 0) under key (seed, scenario_id), words 0-1
// for even q and 2-3 for odd q.  Any sample range can therefore be produced by
// any thread, in any order, with the same result; a call's thread and the
// library's idle sampling threads take [0, n) in pieces of kGrain samples.  Built with -ffp-contract=off so the binary64 transforms
// round the same on every host.
#include <pthread.h>
#include <sched.h>

#include <algorithm>
#include <atomic>
#include <chrono>
#include <cmath>
#include <condition_variable>
#include <cstring>
#include <functional>
#include <list>
#include <mutex>
#include <string>
#include <thread>

#include "aeb_internal.h"
#include "host_util.h"

namespace aeb {
namespace {

inline void mul_hi_lo(uint64_t a, uint64_t b, uint64_t &hi, uint64_t &lo)
{
    const unsigned __int128 p = (unsigned __int128)a * b;
    hi = (uint64_t)(p >> 64);
    lo = (uint64_t)p;
}

// Philox-4x64 with 10 rounds: multipliers 0xD2E7470EE14C6C93, 0xCA5A826395121157,
// Weyl key increments 0x9E3779B97F4A7C15, 0xBB67AE8584CAA73B.
inline void philox4x64_10(uint64_t c[4], uint64_t k0, uint64_t k1)
{
    for (int r = 0; r < 10; ++r) {
        uint64_t h0, l0, h1, l1;
        mul_hi_lo(0xD2E7470EE14C6C93ull, c[0], h0, l0);
        mul_hi_lo(0xCA5A826395121157ull, c[2], h1, l1);
        const uint64_t n0 = h1 ^ c[1] ^ k0, n2 = h0 ^ c[3] ^ k1;
        c[0] = n0;
        c[1] = l1;
        c[2] = n2;
        c[3] = l0;
        k0 += 0x9E3779B97F4A7C15ull;
        k1 += 0xBB67AE8584CAA73Bull;
    }
}

constexpr double kTwoM53 = 1.0 / 9007199254740992.0;

inline double transform(const aeb_dist &d, uint64_t w0, uint64_t w1)
{
    double x;
    switch (d.kind) {
    case AEB_DIST_UNIFORM:
        x = d.p0 + (d.p1 - d.p0) * ((double)(w0 >> 11) * kTwoM53);
        break;
    case AEB_DIST_NORMAL: {
        const double u1 = (double)((w0 >> 11) + 1) * kTwoM53;  // (0, 1]
        const double u2 = (double)(w1 >> 11) * kTwoM53;        // [0, 1)
        x = d.p0 + d.p1 * (std::sqrt(-2.0 * std::log(u1)) * std::cos(6.283185307179586 * u2));
        break;
    }
    default:
        x = d.p0;
    }
    if (x < d.lo) x = d.lo;
    if (x > d.hi) x = d.hi;
    return x;
}

// Importance sampling: probability that an unclamped draw of d lies at or
// below x, or above x.
double mass_below(const aeb_dist &d, double x)
{
    if (d.kind == AEB_DIST_UNIFORM) {
        const double u = (x - d.p0) / (d.p1 - d.p0);
        return u <= 0.0 ? 0.0 : (u >= 1.0 ? 1.0 : u);
    }
    return 0.5 * std::erfc((d.p0 - x) / (d.p1 * std::sqrt(2.0)));
}

double mass_above(const aeb_dist &d, double x)
{
    if (d.kind == AEB_DIST_UNIFORM) return 1.0 - mass_below(d, x);
    return 0.5 * std::erfc((x - d.p0) / (d.p1 * std::sqrt(2.0)));
}

// Likelihood ratio p(x) / q(x) of one quantity drawn from q with clamped
// value x: a clamp bound holding mass under q compares the masses there,
// elsewhere the densities compare.
double likelihood_ratio(const aeb_dist &p, const aeb_dist &q, double x)
{
    if (q.kind == AEB_DIST_CONST) return 1.0;
    if (x <= q.lo) {
        const double mq = mass_below(q, q.lo);
        if (mq > 0.0) return mass_below(p, p.lo) / mq;
    }
    if (x >= q.hi) {
        const double mq = mass_above(q, q.hi);
        if (mq > 0.0) return mass_above(p, p.hi) / mq;
    }
    if (q.kind == AEB_DIST_UNIFORM)
        return (x >= p.p0 && x < p.p1) ? (q.p1 - q.p0) / (p.p1 - p.p0) : 0.0;
    const double zp = (x - p.p0) / p.p1, zq = (x - q.p0) / q.p1;
    return (q.p1 / p.p1) * std::exp(0.5 * (zq * zq - zp * zp));
}

bool is_compatible(const aeb_dist &p, const aeb_dist &q)
{
    if (p.kind != q.kind || p.lo != q.lo || p.hi != q.hi) return false;
    switch (q.kind) {
    case AEB_DIST_CONST: return p.p0 == q.p0;
    case AEB_DIST_UNIFORM: return q.p0 <= p.p0 && p.p1 <= q.p1 && p.p1 > p.p0;
    default: return p.p1 > 0.0 && q.p1 > 0.0;
    }
}

// Samples [lo, hi) of the call; with `nominal`, also their likelihood ratios.
void sample_block(double g, const aeb_scenario &sc, uint64_t first, uint64_t lo, uint64_t hi,
                  const aeb_params &out, const aeb_scenario *nominal, double *weights)
{
    const aeb_dist *dist[9] = {&sc.v0, &sc.d0, &sc.mu, &sc.grade, &sc.mass,
                               &sc.cd, &sc.tau, &sc.t_delay, &sc.noise};
    const aeb_dist *ndist[9] = {};
    if (nominal) {
        const aeb_dist *nd[9] = {&nominal->v0, &nominal->d0, &nominal->mu, &nominal->grade,
                                 &nominal->mass, &nominal->cd, &nominal->tau,
                                 &nominal->t_delay, &nominal->noise};
        for (int q = 0; q < 9; ++q) ndist[q] = nd[q];
    }
    for (uint64_t j = lo; j < hi; ++j) {
        double q[10];
        for (uint64_t b = 0; b < 5; ++b) {
            uint64_t c[4] = {first + j, b, 0, 0};
            philox4x64_10(c, sc.seed, sc.scenario_id);
            q[2 * b] = transform(*dist[2 * b], c[0], c[1]);
            if (2 * b + 1 < 9) q[2 * b + 1] = transform(*dist[2 * b + 1], c[2], c[3]);
        }
        out.v0[j] = q[0];
        out.d0[j] = q[1];
        out.mu[j] = q[2];
        out.gs[j] = g * std::sin(q[3]);
        out.gc[j] = g * std::cos(q[3]);
        out.mass[j] = q[4];
        out.cd[j] = q[5];
        out.tau[j] = q[6];
        out.t_delay[j] = q[7];
        out.noise[j] = q[8];
        if (nominal) {
            double w = 1.0;
            for (int k = 0; k < 9; ++k) w *= likelihood_ratio(*ndist[k], *dist[k], q[k]);
            weights[j] = w;
        }
    }
}

bool dist_ok(const aeb_dist &d)
{
    if (d.reserved != 0) return false;
    if (d.kind != AEB_DIST_CONST && d.kind != AEB_DIST_UNIFORM && d.kind != AEB_DIST_NORMAL)
        return false;
    if (!std::isfinite(d.p0) || !std::isfinite(d.p1)) return false;
    if (std::isnan(d.lo) || std::isnan(d.hi) || d.lo > d.hi) return false;
    return true;
}

// Samples a piece takes on one thread (~170 ns each): ~45 us, a few times what
// waking a thread costs.
constexpr uint64_t kGrain = 256;

// Sampling threads shared by every call of the process.  Starting and joining
// 16 threads takes ~1 ms, more than sampling 50,000 samples on them; these are
// started when a call first wants them (one fewer than the host's threads), wait
// for work and end after a second without any.  The calling thread works too
// and only waits for pieces a helper has begun, so a call never depends on a
// helper being there.  A helper runs on the CPUs of the call it helps (as a thread
// that the call had started would), not on those of the call that started it.
class Workers {
  public:
    using Piece = std::function<void(uint64_t, uint64_t)>;

    static Workers &get()
    {
        static std::once_flag once;
        std::call_once(once, [] {
            instance() = new Workers;  // never destroyed: helpers may outlive static objects
            // a forked child has none of the parent's threads
            pthread_atfork(nullptr, nullptr, [] { instance() = new Workers; });
        });
        return *instance();
    }

    // f over [0, n) in pieces, on at most `threads` threads, this one included.
    void run(uint64_t n, unsigned threads, const Piece &f)
    {
        Job job(n, &f, threads > 0 ? threads - 1 : 0);
        const uint64_t pieces = (n + kGrain - 1) / kGrain;
        const unsigned helpers =
            (unsigned)std::min<uint64_t>({job.max_helpers, pieces - 1, max_threads_});
        if (helpers > 0) {
            job.note_cpus();
            std::lock_guard<std::mutex> lk(mu_);
            jobs_.push_back(&job);
            while (idle_ + starting_ < helpers && threads_ < max_threads_) {
                try {
                    std::thread([this] { loop(); }).detach();
                } catch (...) {
                    break;  // fewer helpers
                }
                ++threads_;
                ++starting_;
            }
            work_.notify_all();
        }
        job.take();
        if (helpers > 0) {
            std::unique_lock<std::mutex> lk(mu_);
            jobs_.remove(&job);
            done_.wait(lk, [&] { return job.helpers == 0; });
        }
    }

  private:
    struct Job {
        const uint64_t n;
        const Piece *f;
        const unsigned max_helpers;
        std::atomic<uint64_t> next{0};
        unsigned helpers = 0;  // threads inside take(), under the pool's lock
        cpu_set_t cpus;        // of the calling thread (cpus_known)
        bool cpus_known = false;
        Job(uint64_t n_, const Piece *f_, unsigned m) : n(n_), f(f_), max_helpers(m) {}
        void note_cpus()
        {
            cpus_known = pthread_getaffinity_np(pthread_self(), sizeof cpus, &cpus) == 0;
        }
        void take()
        {
            for (uint64_t lo; (lo = next.fetch_add(kGrain)) < n;)
                (*f)(lo, std::min(n, lo + kGrain));
        }
    };

    static Workers *&instance()
    {
        static Workers *w = nullptr;
        return w;
    }

    void loop()
    {
        cpu_set_t mine;
        bool known = pthread_getaffinity_np(pthread_self(), sizeof mine, &mine) == 0;
        std::unique_lock<std::mutex> lk(mu_);
        --starting_;
        for (;;) {
            Job *job = nullptr;
            for (Job *j : jobs_)
                if (j->helpers < j->max_helpers && j->next.load() < j->n) {
                    job = j;
                    break;
                }
            if (!job) {
                ++idle_;
                const auto r = work_.wait_for(lk, std::chrono::seconds(1));
                --idle_;
                if (r == std::cv_status::timeout && jobs_.empty()) {
                    --threads_;
                    return;
                }
                continue;
            }
            ++job->helpers;
            lk.unlock();
            if (job->cpus_known && !(known && CPU_EQUAL(&mine, &job->cpus))) {
                mine = job->cpus;
                known = pthread_setaffinity_np(pthread_self(), sizeof mine, &mine) == 0;
            }
            job->take();
            lk.lock();
            if (--job->helpers == 0) done_.notify_all();  // the job may be gone after this
        }
    }

    std::mutex mu_;
    std::condition_variable work_, done_;
    std::list<Job *> jobs_;
    unsigned threads_ = 0, idle_ = 0, starting_ = 0;
    const unsigned max_threads_ = std::max(2u, std::thread::hardware_concurrency()) - 1;
};

unsigned sampling_threads(int32_t n_threads)
{
    const unsigned hw = std::thread::hardware_concurrency();
    return n_threads > 0 ? (unsigned)n_threads : (hw ? hw : 1);
}

}  // namespace
}  // namespace aeb

namespace aeb {
namespace {

aeb_status sample_impl(const char *who, const aeb_model *model, const aeb_scenario *scenario,
                       const aeb_scenario *nominal, uint64_t first, uint64_t n,
                       const aeb_params *out, double *weights, int32_t n_threads)
{
    const std::string w = who;
    if (!model || !scenario || !out) return fail(AEB_EINVAL, w + ": NULL argument");
    if (!std::isfinite(model->g)) return fail(AEB_EINVAL, w + ": g is not finite");
    const aeb_dist *dist[9] = {&scenario->v0, &scenario->d0, &scenario->mu, &scenario->grade,
                               &scenario->mass, &scenario->cd, &scenario->tau,
                               &scenario->t_delay, &scenario->noise};
    for (int q = 0; q < 9; ++q)
        if (!dist_ok(*dist[q]))
            return fail(AEB_EINVAL, w + ": invalid distribution for quantity " + std::to_string(q));
    if (nominal) {
        if (!weights) return fail(AEB_EINVAL, w + ": NULL weights");
        const aeb_dist *nd[9] = {&nominal->v0, &nominal->d0, &nominal->mu, &nominal->grade,
                                 &nominal->mass, &nominal->cd, &nominal->tau,
                                 &nominal->t_delay, &nominal->noise};
        for (int q = 0; q < 9; ++q)
            if (!dist_ok(*nd[q]) || !is_compatible(*nd[q], *dist[q]))
                return fail(AEB_EINVAL, w + ": proposal incompatible with the nominal scenario "
                                            "for quantity " + std::to_string(q));
    }
    if (n == 0) return AEB_OK;
    const double *cols[AEB_NFIELDS] = {out->v0, out->d0, out->mu, out->gs, out->gc,
                                       out->mass, out->cd, out->tau, out->t_delay, out->noise};
    for (int j = 0; j < AEB_NFIELDS; ++j)
        if (!cols[j]) return fail(AEB_EINVAL, w + ": NULL output column");

    const aeb_scenario sc = *scenario;
    const aeb_params o = *out;
    Workers::get().run(n, sampling_threads(n_threads), [&](uint64_t lo, uint64_t hi) {
        sample_block(model->g, sc, first, lo, hi, o, nominal, weights);
    });
    return AEB_OK;
}

}  // namespace

void sample_scenarios(const aeb_model &model, const aeb_scenario *scenarios, uint32_t n_scen,
                      uint64_t n_per, const aeb_params &out)
{
    const auto piece = [&](uint64_t lo, uint64_t hi) {
        while (lo < hi) {  // the part of [lo, hi) in one scenario
            const uint64_t sc = lo / n_per, base = sc * n_per, end = std::min(hi, base + n_per);
            aeb_params o = out;
            double **c[AEB_NFIELDS] = {&o.v0, &o.d0, &o.mu, &o.gs, &o.gc,
                                       &o.mass, &o.cd, &o.tau, &o.t_delay, &o.noise};
            for (auto p : c) *p += base;
            sample_block(model.g, scenarios[sc], 0, lo - base, end - base, o, nullptr, nullptr);
            lo = end;
        }
    };
    Workers::get().run(n_scen * n_per, sampling_threads(0), piece);
}

}  // namespace aeb

extern "C" aeb_status aeb_sample_params(const aeb_model *model, const aeb_scenario *scenario,
                                        uint64_t first, uint64_t n, const aeb_params *out,
                                        int32_t n_threads)
{
    aeb::clear_error();
    return aeb::sample_impl("aeb_sample_params", model, scenario, nullptr, first, n, out,
                            nullptr, n_threads);
}

extern "C" aeb_status aeb_sample_params_is(const aeb_model *model, const aeb_scenario *nominal,
                                           const aeb_scenario *proposal, uint64_t first,
                                           uint64_t n, const aeb_params *out, double *weights,
                                           int32_t n_threads)
{
    aeb::clear_error();
    if (!nominal) return aeb::fail(AEB_EINVAL, "aeb_sample_params_is: NULL nominal scenario");
    return aeb::sample_impl("aeb_sample_params_is", model, proposal, nominal, first, n, out,
                            weights, n_threads);
}
