// rollout_fp64.cu -- binary64 rollout kernel, bit-identical to the plain
// definition of the method.
//
// Build: -fmad=false, so no multiply and add pair is ever fused; every
// expression below is evaluated in the order written, with IEEE round-to-
// nearest division.  The per-sample constants, the RK4 stages (Sec. IV-D,
// Eq. 7-9), the realised deceleration (Eq. 4-5 / per-axle caps), the command
// schedule, the termination tests (Sec. V-D) and the refinement are written
// in the same operation order as the binary64 definition, so each output is
// the same bits (Sec. V-D: same samples, same integrator, same precision,
// same termination, no fused or approximate operations).
//
// The realised deceleration is the minimum of lines (D, mu g cos(theta) and
// the two axle lines, or D and the Eq. 5 cap), and a minimum returns one of
// its arguments unchanged.  So a lane keeps the line that is the strict
// minimum over an interval [dlo, dhi] of demand, shrunk at each end by a band
// of 1e-12 relative (far above the few-ulp rounding of a line value, so no
// rounding can change which line is smallest inside it); while a step's
// stage demands lie in the interval (the first stage has the smallest demand
// and the fourth the largest when dt / tau <= 2), each stage evaluates only
// that line, with the same expression as the full minimum, and the result
// is the same bits.  Other steps evaluate the full minimum and re-select.
//
// What bounds it.  An SM sub-partition's binary64 unit holds a warp
// instruction for 64 cycles if it is a fused multiply-add of three register
// operands and for 76 otherwise (an add, a multiply, an immediate or constant
// operand), whatever the number of warps, chains or busy lanes.  So inside a
// piece every operation is written as a fused multiply-add of registers that
// rounds to the same bits: a + b is fma(a, 1, b), a b is fma(a, b, -0), and
// v + 2 w is fma(2, w, v), since doubling is exact away from overflow (a lane
// takes this path only while its state is far inside the normal range, see
// `tame`); the constants 1, 2, -0, dt and its fractions are kept in registers
// the compiler cannot take for constants.  51 operations of 64 cycles a step
// (59 on an axle line) against 57 (65) of 76.
//
// A rollout spends most of its steps where r(D) cannot change: before brake
// onset (a = u = 0), and after it once the demand is on the constant cap, which
// a growing demand never leaves (icy and wet roads; about half of the
// single-scenario workload's steps), or with an instantaneous actuator.  A
// warp whose lanes are all there runs a step without the actuator and with r
// held: 32 operations (27 and the position) instead of 51.  order.cu hands a
// warp samples of one cap class and length, so that its lanes are there
// together.
#include <climits>

#include "rollout_common.cuh"

namespace aeb {
namespace {

__device__ __forceinline__ double dmin(double a, double b) { return (b < a) ? b : a; }

// The per-step comparisons as integer comparisons of the bit patterns (the
// binary64 pipe is the narrow one here): each gives the same truth value as
// the binary64 comparison it replaces.

// x <= 0.0 (false for a NaN).
__device__ __forceinline__ bool le_zero(double x)
{
    const int hi = __double2hiint(x), lo = __double2loint(x);
    const unsigned mag = (unsigned)hi & 0x7fffffffu;
    const bool nan = mag > 0x7ff00000u || (mag == 0x7ff00000u && lo != 0);
    return !nan && (hi < 0 || (mag | (unsigned)lo) == 0u);
}

// x >= y for a finite y > 0 (false for a NaN x): non-negative doubles order
// as their bit patterns, and every negative x (-0 included) has the sign bit.
__device__ __forceinline__ bool ge_pos(double x, double y)
{
    const long long bx = __double_as_longlong(x), by = __double_as_longlong(y);
    return bx >= by && bx <= 0x7ff0000000000000ll;
}

// Order key of a non-NaN double: a signed integer that increases with the
// value and is equal for -0 and +0; okey(-x) = -okey(x).
__device__ __forceinline__ long long okey(double x)
{
    const long long b = __double_as_longlong(x);
    return b < 0 ? -(b & 0x7fffffffffffffffll) : b;
}

// int_to_double(n) for n >= 0, exact, on the integer pipe.
__device__ __forceinline__ double from_int(int32_t n)
{
    if (n <= 0) return 0.0;
    const int e = 31 - __clz(n);
    const long long m = (long long)n << (52 - e);  // implicit one at bit 52
    return __longlong_as_double(m + ((long long)(1022 + e) << 52));
}

// Step constants in registers, and the operations of a step as fused
// multiply-adds of register operands (the same bits as the plain operation).
struct Ops {
    double one, two, nz, dt, h2, h6;
    __device__ __forceinline__ double add(double a, double b) const { return __fma_rn(a, one, b); }
    __device__ __forceinline__ double sub(double a, double b) const { return __fma_rn(b, -one, a); }
    __device__ __forceinline__ double mul(double a, double b) const { return __fma_rn(a, b, nz); }
    // a + 2 b, where 2 b does not overflow
    __device__ __forceinline__ double add2(double a, double b) const { return __fma_rn(two, b, a); }
    // h6 (((a + 2 b) + 2 c) + d) + y, rounded after each operation of the definition
    __device__ __forceinline__ double combine(double y, double a, double b, double c, double d) const
    {
        return add(y, mul(h6, add(add2(add2(a, b), c), d)));
    }
};

// Bounds of the states the fused forms are used on: they keep every sum and
// product of a step below 2^400, so nothing overflows.
constexpr int kTtcSpan = 256;  // steps one trigger test may cover
constexpr double kTame = 1e5;
__device__ __forceinline__ bool tame_speed(double v)  // 0 < v < ~1e5 (false for a NaN)
{
    return (unsigned)__double2hiint(v) < 0x40f86a00u;
}

__device__ __forceinline__ double dinf() { return __longlong_as_double(0x7ff0000000000000ll); }

// Moving lead (extension): the lead brakes from lead_v0 at lead_decel until it
// stops (stop time lead_ts, stop position lead_xs), in closed form.
__device__ __forceinline__ double lead_pos(const ModelDev &M, double t)
{
    if (M.lead_decel > 0.0 && t >= M.lead_ts) return M.lead_xs;
    return t * (M.lead_v0 - (0.5 * M.lead_decel) * t);
}

__device__ __forceinline__ double lead_speed(const ModelDev &M, double t)
{
    if (M.lead_decel > 0.0 && t >= M.lead_ts) return 0.0;
    return M.lead_v0 - M.lead_decel * t;
}

template <int CAP, bool LEAD, bool TTC>
struct Lane64 {
    double x, v, a;
    double d0, gs, noise, k, it, thr;
    double mg, f0, f1, r0, r1, cap;
    double pa, pb;                // current line pa + pb D (piece 1, 2)
    long long klo, khi;           // its demand interval [dlo, dhi] as order keys
    uint64_t row;                 // perception key row (counter of the readings)
    int32_t n, n_b, n_delay;
    int piece;                    // 0: D, 1, 2: an axle line, 3: the constant cap; -1: none
    bool trig, lagged, ordered;
    bool active;                  // the lane holds a rollout
    bool damped;                  // dt / tau <= 1: the stage demands approach -a_cmd from below
    bool held;                    // r is the same at every stage until onset, or for good
    double nr;                    // -r while held
    int32_t n_chk;                // TTC: no step before this one can trigger

    // Select the line that is the strict minimum at demand D and the demand
    // interval, shrunk by the band, on which it stays so (piece -1 if D is
    // inside a band, lines are nearly parallel, or the stage demands are not
    // ordered).
    __device__ void select_piece(double D)
    {
        piece = -1;
        if (!ordered) return;
        double A[4], S[4];
        int nl;
        if (CAP == AEB_CAP_LUMPED) {
            A[0] = 0.0; S[0] = 1.0; A[1] = cap; S[1] = 0.0;
            nl = 2;
        } else {
            A[0] = 0.0; S[0] = 1.0; A[1] = f0; S[1] = f1; A[2] = r0; S[2] = r1; A[3] = mg; S[3] = 0.0;
            nl = 4;
        }
        double val[4];
        int cur = 0;
        for (int j = 0; j < nl; ++j) {
            val[j] = (j == 0) ? D : A[j] + S[j] * D;
            if (val[j] < val[cur]) cur = j;
        }
        double lo = -dinf(), hi = dinf();
        for (int j = 0; j < nl; ++j) {
            if (j == cur) continue;
            const double ds = S[cur] - S[j];
            if (!(fabs(ds) >= 1e-6) || !(val[j] > val[cur])) return;
            const double B = (A[j] - A[cur]) / ds;  // line j meets the current line
            const double band = 1e-12 * (1.0 + fabs(A[j]) + fabs(A[cur]) + fabs(B)) / fabs(ds);
            if (ds > 0.0) hi = fmin(hi, B - band);  // line j is below beyond B
            else lo = fmax(lo, B + band);
        }
        if (!(lo <= D && D <= hi)) return;
        if (!(fabs(A[cur]) < 1e50 && fabs(S[cur]) < 1e50)) return;  // see Ops
        klo = okey(lo);
        khi = okey(hi);
        if (CAP == AEB_CAP_LUMPED) {
            piece = (cur == 0) ? 0 : 3;
        } else {
            piece = cur;
            pa = A[cur];
            pb = S[cur];
        }
    }

    // dv/dt on the current piece: the same value as `accel` for D in the
    // piece's interval.  `lines`: some lane of the warp is on an axle line.
    __device__ __forceinline__ double accel_piece(const Ops &q, double vv, double aa,
                                                  bool lines) const
    {
        const double D = -aa;
        const double c = (CAP == AEB_CAP_LUMPED) ? cap : mg;
        double r = (piece == 0) ? D : c;
        if (CAP != AEB_CAP_LUMPED && lines) {
            const double rl = q.add(pa, q.mul(pb, D));
            if (piece == 1 || piece == 2) r = rl;
        }
        return q.sub(q.sub(-r, q.mul(q.mul(k, vv), vv)), gs);
    }

    // Realised deceleration r for demand D = -a (Eq. 5 as printed, or the
    // per-axle fixed point min(min(D, mu gc), min(f0 + f1 D, r0 + r1 D))),
    // then dv/dt = -r - k v^2 - g sin(theta) (Eq. 4).
    __device__ __forceinline__ double realised(double D) const
    {
        if (CAP == AEB_CAP_LUMPED) return dmin(D, cap);
        double lf = f0 + f1 * D;
        double lr = r0 + r1 * D;
        return dmin(dmin(D, mg), dmin(lf, lr));
    }
    __device__ __forceinline__ double accel(double vv, double aa) const
    {
        const double r = realised(-aa);
        return ((-r) - (k * vv) * vv) - gs;
    }

    // Hold r at the actuator value aa, at which the lane stays until onset (0)
    // or for good (an instantaneous actuator's command).
    __device__ __forceinline__ void hold_at(double aa)
    {
        held = ordered;
        nr = -realised(-aa);
    }

    // After a step inside a piece, braking: whether the lane is on the constant
    // cap for good.  The stage demands of a damped lag lie between the present
    // demand and -a_cmd up to a few ulps (and so do all later ones), and the
    // constant stays the strict minimum above klo, so it is enough that the
    // present demand is 2^12 ulps above klo (a positive value) and a >= a_cmd.
    __device__ __forceinline__ void try_hold(const ModelDev &M)
    {
        if (piece == 3 && damped && khi == 0x7ff0000000000000ll &&
            klo > 0x3f50000000000000ll /* 2^-10 */ && -okey(a) >= klo + 4096 &&
            okey(a) >= okey(M.a_cmd)) {
            held = true;
            nr = (CAP == AEB_CAP_LUMPED) ? -cap : -mg;
        }
    }

    __device__ __forceinline__ int32_t onset() const
    {
        return TTC ? (trig ? n_b : -1) : n_delay;
    }

    __device__ __forceinline__ bool init(const ModelDev &M, const ParamsDev &P,
                                         const OutDev &O, const Row &rows)
    {
        double f[AEB_NFIELDS];
        const uint64_t i = rows.o;
        load_fields(P, rows.p, f);
        thr = rows.thr;
        if (!sample_valid(f)) {
            const double nan = __longlong_as_double(0x7ff8000000000000ll);
            store_out(O, i, AEB_INVALID, nan, nan, nan, nan, 0, -1);
            return true;
        }
        row = rows.k;
        d0 = f[kD0];
        gs = f[kGs];
        noise = f[kNoise];
        k = ((M.rho * f[kCd]) * M.area) / (2.0 * f[kMass]);
        lagged = f[kTau] > 0.0;
        it = lagged ? 1.0 / f[kTau] : 0.0;
        // (and the sample is inside the range of the fused forms)
        ordered = (!lagged || M.dt * it <= 2.0) && M.dt >= 1e-30 && M.dt <= 1.0 &&
                  fabs(M.a_cmd) <= kTame && k <= 1.0 && fabs(gs) <= kTame;
        damped = lagged && M.dt * it <= 1.0 && M.a_cmd < 0.0;
        const double mu = f[kMu], gc = f[kGc];
        const double mh = mu * M.hl;
        if (CAP == AEB_CAP_LUMPED) {
            cap = (mu * M.g) / (1.0 + mh);
        } else {
            mg = mu * gc;
            f0 = (mg * M.phi_f) / (1.0 - mh);
            f1 = (1.0 - M.beta) / (1.0 - mh);
            r0 = (mg * (1.0 - M.phi_f)) / (1.0 + mh);
            r1 = M.beta / (1.0 + mh);
        }
        n_delay = steps_to_reach_dev(f[kTdelay], M.dt);
        trig = !TTC;
        n_b = n_delay;
        const int32_t on = TTC ? -1 : n_delay;
        if (LEAD && d0 <= 0.0) {
            store_out(O, i, AEB_CONTACT, 0.0, 0.0, f[kV0], 0.0, 0, on);
            return true;
        }
        if (f[kV0] <= 0.0) {
            store_out(O, i, AEB_STOP, 0.0, 0.0, 0.0, 0.0, 0, on);
            return true;
        }
        if (M.n_max == 0) {
            store_out(O, i, AEB_HORIZON, 0.0, 0.0, 0.0, 0.0, 0, on);
            return true;
        }
        x = 0.0;
        v = f[kV0];
        a = 0.0;
        n = 0;
        n_chk = 0;
        select_piece(-a);
        hold_at(a);
        return false;
    }

    // TTC trigger (while not yet triggered), at the start of step n.  A test
    // that does not fire also bounds the steps that cannot (n_chk): while r is
    // held the car's acceleration is at most acc = max(0, -r - g sin(theta)),
    // so over kTtcSpan steps its speed stays below W = v + kTtcSpan dt acc and
    // the margin (gap + noise) - thr c falls by at most dt (W + |thr| (acc + b_L))
    // per step (a braking lead's travel only widens the gap; its speed falls by
    // dt b_L); a reading's noise is at most 3 perc_sigma.
    __device__ __forceinline__ void test_trigger(const ModelDev &M, const Ops &q)
    {
        double gap_meas, closing;
        if (M.lead_moving) {  // gap and closing speed to the moving lead
            const double t = from_int(n) * q.dt;
            gap_meas = ((d0 + lead_pos(M, t)) - x) + noise;
            closing = v - lead_speed(M, t);
        } else {
            gap_meas = q.add(q.sub(d0, x), noise);
            closing = v;
        }
        const double limit = q.mul(thr, closing);
        const float margin = (float)(gap_meas - limit) - 3.001f * (float)M.perc_sigma;
        bool reading = true;
        if (M.perc && !(margin > 0.0f)) {  // the reading of step n + L describes step n
            uint32_t h[4];
            perc_halves(row, (uint64_t)((long long)n + M.perc_lat), M.perc_seed, h);
            const double s32 = 1.0 / 4294967296.0;  // 2^-32
            const double u1 = (double)h[0] * s32, u2 = (double)h[1] * s32;
            const double u3 = (double)h[2] * s32, u4 = (double)h[3] * s32;
            if (u4 < M.perc_drop) reading = false;
            else gap_meas = gap_meas + M.perc_sigma * (2.0 * (((u1 + u2) + u3) - 1.5));
        }
        if (reading && gap_meas <= limit) {
            trig = true;
            long long nb = ((long long)n + M.perc_lat) + n_delay;
            n_b = nb > INT_MAX ? INT_MAX : (int32_t)nb;
        } else if (held && margin > 0.0f && tame_speed(v)) {
            const float dtf = (float)q.dt, acc = fmaxf(0.0f, (float)(nr - gs));
            const float W = (float)v + (float)kTtcSpan * dtf * acc;
            const float fall = dtf * (W + fabsf((float)thr) * (acc + (float)M.lead_decel)) * 1.001f;
            // margin's own rounding: a few binary32 ulps of what it was formed from
            const float m = margin * 0.999f - 1e-5f * (fabsf((float)gap_meas) + fabsf((float)limit));
            const float steps = __fdividef(m, fall);
            if (steps > 1.0f) n_chk = n + (steps < (float)kTtcSpan ? (int)steps : kTtcSpan);
        }
    }

    // One RK4 step (all lanes of the warp together); true if the lane's rollout
    // ended (stored).
    __device__ __forceinline__ bool step(const ModelDev &M, const Ops &q, const OutDev &O,
                                         uint64_t i)
    {
        const double dt = q.dt, h2 = q.h2, h6 = q.h6;
        if (TTC && active && !trig && n >= n_chk) test_trigger(M, q);
        if (trig && n == n_b) {  // the command switches on: a moves from here, or has moved
            held = false;
            if (!lagged) hold_at(M.a_cmd);
        }
        const bool braking = trig && n >= n_b;
        const double u = braking ? M.a_cmd : 0.0;
        double v2, v3, v4, xn, vn, an;
        bool pw = true;
        if (__all_sync(kFull, !active || (held && tame_speed(v)))) {
            const double kv1 = q.sub(q.sub(nr, q.mul(q.mul(k, v), v)), gs);
            v2 = q.add(v, q.mul(h2, kv1));
            const double kv2 = q.sub(q.sub(nr, q.mul(q.mul(k, v2), v2)), gs);
            v3 = q.add(v, q.mul(h2, kv2));
            const double kv3 = q.sub(q.sub(nr, q.mul(q.mul(k, v3), v3)), gs);
            v4 = q.add(v, q.mul(dt, kv3));
            const double kv4 = q.sub(q.sub(nr, q.mul(q.mul(k, v4), v4)), gs);
            xn = q.combine(x, v, v2, v3, v4);
            vn = q.combine(v, kv1, kv2, kv3, kv4);
            an = lagged ? a : u;  // not read while r is held
        } else {
            double a1, a2, a3, a4, ka1 = 0.0, ka2 = 0.0, ka3 = 0.0, ka4 = 0.0;
            if (lagged) {
                a1 = a;
                ka1 = q.mul(q.sub(u, a1), it);
                a2 = q.add(a, q.mul(h2, ka1));
                ka2 = q.mul(q.sub(u, a2), it);
                a3 = q.add(a, q.mul(h2, ka2));
                ka3 = q.mul(q.sub(u, a3), it);
                a4 = q.add(a, q.mul(dt, ka3));
                ka4 = q.mul(q.sub(u, a4), it);
            } else {
                a1 = a2 = a3 = a4 = u;
            }
            // With dt / tau <= 2 the stage demands lie between the first and the
            // fourth (-a1 smallest when the command is a deceleration, so that
            // a - u >= 0 from the start, -a4 smallest otherwise): two tests for
            // the step.
            // (A piece exists only when dt / tau <= 2, where the lag is stable and
            // the stage actuator values are finite, so order keys compare them.)
            const bool dec = M.a_cmd <= 0.0;
            const long long kfirst = -okey(dec ? a1 : a4), klast = -okey(dec ? a4 : a1);
            pw = piece >= 0 && kfirst >= klo && klast <= khi && tame_speed(v);
            const bool lines = __any_sync(kFull, active && pw && (piece == 1 || piece == 2));
            if (pw) {
                const double kv1 = accel_piece(q, v, a1, lines);
                v2 = q.add(v, q.mul(h2, kv1));
                const double kv2 = accel_piece(q, v2, a2, lines);
                v3 = q.add(v, q.mul(h2, kv2));
                const double kv3 = accel_piece(q, v3, a3, lines);
                v4 = q.add(v, q.mul(dt, kv3));
                const double kv4 = accel_piece(q, v4, a4, lines);
                xn = q.combine(x, v, v2, v3, v4);
                vn = q.combine(v, kv1, kv2, kv3, kv4);
                an = lagged ? q.combine(a, ka1, ka2, ka3, ka4) : u;
            } else if (active) {
                const double kv1 = accel(v, a1);
                v2 = v + h2 * kv1;
                const double kv2 = accel(v2, a2);
                v3 = v + h2 * kv2;
                const double kv3 = accel(v3, a3);
                v4 = v + dt * kv3;
                const double kv4 = accel(v4, a4);
                xn = x + h6 * (((v + 2.0 * v2) + 2.0 * v3) + v4);
                vn = v + h6 * (((kv1 + 2.0 * kv2) + 2.0 * kv3) + kv4);
                an = lagged ? a + h6 * (((ka1 + 2.0 * ka2) + 2.0 * ka3) + ka4) : u;
            }
        }
        if (!active) return false;

        if (LEAD && M.lead_moving) {
            const double t0 = from_int(n) * dt, t1 = from_int(n + 1) * dt;
            const double g1 = (d0 + lead_pos(M, t1)) - xn;
            if (g1 <= 0.0) {
                const double g0 = (d0 + lead_pos(M, t0)) - x;
                const double c0 = v - lead_speed(M, t0), c1 = vn - lead_speed(M, t1);
                const double s = g0 / (g0 - g1);
                store_out(O, i, AEB_CONTACT, xn, x + s * (xn - x), c0 + s * (c1 - c0),
                          ((double)n + s) * dt, n + 1, onset());
                return true;
            }
        } else if (LEAD && ge_pos(xn, d0)) {  // d0 > 0 and finite here
            const double s = (d0 - x) / (xn - x);
            store_out(O, i, AEB_CONTACT, xn, d0, v + s * (vn - v), ((double)n + s) * dt, n + 1,
                      onset());
            return true;
        }
        if (le_zero(vn)) {
            const double s = v / (v - vn);
            store_out(O, i, AEB_STOP, xn, x + s * (xn - x), 0.0, ((double)n + s) * dt, n + 1,
                      onset());
            return true;
        }
        if (n + 1 >= M.n_max) {
            store_out(O, i, AEB_HORIZON, xn, xn, 0.0, (double)(n + 1) * dt, n + 1, onset());
            return true;
        }
        x = xn;
        v = vn;
        a = an;
        n = n + 1;
        if (!pw) select_piece(-a);
        else if (braking && !held) try_hold(M);
        return false;
    }
};

#ifndef AEB_FP64_MIN_BLOCKS
#define AEB_FP64_MIN_BLOCKS 1  // resident blocks per SM the register budget must allow
#endif

template <int CAP, bool LEAD, bool TTC>
__global__ void __launch_bounds__(128, AEB_FP64_MIN_BLOCKS)
k_rollout_fp64(ModelDev M, ParamsDev P, OutDev O, WorkDev W)
{
    // Each lane owns one rollout at a time (Sec. V-A, one thread per sample); a
    // lane whose rollout ends takes the next sample of its warp's ticket, so a
    // warp keeps its lanes busy until the tickets run out instead of idling
    // until its slowest rollout ends.  There is no wait on other warps or on
    // the host: the loop ends when no lane holds a rollout.
    __shared__ double cst[6][128];
    cst[0][threadIdx.x] = 1.0;
    cst[1][threadIdx.x] = 2.0;
    cst[2][threadIdx.x] = -0.0;
    cst[3][threadIdx.x] = M.dt;
    cst[4][threadIdx.x] = M.h2;
    cst[5][threadIdx.x] = M.h6;
    __syncthreads();  // (read back per lane: register operands, see above)
    const unsigned t = threadIdx.x ^ (unsigned)(W.n >> 63);
    const Ops q{cst[0][t], cst[1][t], cst[2][t], cst[3][t], cst[4][t], cst[5][t]};
    const unsigned lane = threadIdx.x & 31u;
    WarpQueue wq;
    Lane64<CAP, LEAD, TTC> L;
    L.active = false;
    L.x = L.v = L.a = L.d0 = L.gs = L.noise = L.k = L.it = L.thr = 0.0;
    L.mg = L.f0 = L.f1 = L.r0 = L.r1 = L.cap = L.pa = L.pb = 0.0;
    L.klo = L.khi = 0;
    L.row = 0;
    L.n = L.n_b = L.n_delay = 0;
    L.piece = -1;
    L.trig = L.lagged = L.ordered = L.damped = L.held = false;
    L.nr = 0.0;
    L.n_chk = 0;
    uint64_t oidx = 0;
    unsigned need = kFull;
    for (;;) {
        while (need) {
            uint32_t pos = 0;
            const bool got = wq.take(need, W, pos);
            bool ended = false;
            if ((need >> lane) & 1u) {
                L.active = got;
                if (got) {
                    const Row rows = row_of(W, pos, M.ttc_thr);
                    oidx = rows.o;
                    ended = L.init(M, P, O, rows);
                }
            }
            need = __ballot_sync(kFull, ended);
        }
        if (!__any_sync(kFull, L.active)) return;
        need = __ballot_sync(kFull, L.step(M, q, O, oidx));
    }
}

template <int CAP, bool LEAD, bool TTC>
cudaError_t launch_t(const ModelDev &m, const ParamsDev &p, const OutDev &o, const WorkDev &w,
                     const LaunchCfg &cfg, cudaStream_t s)
{
    auto kern = k_rollout_fp64<CAP, LEAD, TTC>;
    int dev = 0, sms = 0, per_sm = cfg.blocks_per_sm;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    if (per_sm <= 0) {
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, 128, 0);
        if (e != cudaSuccess) return e;
        if (per_sm < 1) per_sm = 1;
    }
    uint64_t blocks = (uint64_t)sms * per_sm;
    const uint64_t need_blocks = (tickets_of(w) + 3) / 4;  // one ticket per warp at least
    if (need_blocks < blocks) blocks = need_blocks;
    if (blocks < 1) blocks = 1;
    kern<<<(unsigned)blocks, 128, 0, s>>>(m, p, o, w);
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_rollout_fp64(const ModelDev &m, const ParamsDev &p, const OutDev &o,
                                const WorkDev &w, const LaunchCfg &cfg, cudaStream_t s)
{
    const bool lead = m.lead != 0, ttc = m.trigger == AEB_TRIGGER_TTC;
    if (m.cap_mode == AEB_CAP_LUMPED) {
        if (lead) return ttc ? launch_t<AEB_CAP_LUMPED, true, true>(m, p, o, w, cfg, s)
                             : launch_t<AEB_CAP_LUMPED, true, false>(m, p, o, w, cfg, s);
        return ttc ? launch_t<AEB_CAP_LUMPED, false, true>(m, p, o, w, cfg, s)
                   : launch_t<AEB_CAP_LUMPED, false, false>(m, p, o, w, cfg, s);
    }
    if (lead) return ttc ? launch_t<AEB_CAP_PER_AXLE, true, true>(m, p, o, w, cfg, s)
                         : launch_t<AEB_CAP_PER_AXLE, true, false>(m, p, o, w, cfg, s);
    return ttc ? launch_t<AEB_CAP_PER_AXLE, false, true>(m, p, o, w, cfg, s)
               : launch_t<AEB_CAP_PER_AXLE, false, false>(m, p, o, w, cfg, s);
}

}  // namespace aeb
