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
//
// The unit can be relieved further: its 64 cycles hold 64 issue slots, of which
// a binary64 multiply or add in integer arithmetic (soft64.h) takes 20-25.  So
// when a launch fills the GPU, the products and the additions of a small
// increment to a large value (30 of 51 operations, 18 of 32) run on the integer
// pipes beside the unit, each the same bits; a step in which one does not apply
// (a zero, a sum three binades away; ~4 % of a warp's steps) is taken again on
// the unit.  1e6 rollouts 262 -> 169 ms, 250,007 69 -> 48 ms.  Bound by latency
// and issue: per warp step ~24 operations on the unit (75 % busy), ~670 on the
// half-rate integer pipe (65 %).  The stages run as a loop: unrolled, the step's
// 20 KB of code wait on the instruction caches (+6 %).
//
// Steps run in runs (Lane64::run) with no event test inside, each step's state
// tested while the next is computed: a warp alone took 2,740 cycles for a held
// step and 4,540 for another, now 2,300 (2,048 on the unit) and 3,850.
#include <climits>

#include "rollout_common.cuh"
#include "soft64.h"

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

// The step constants as factors of software multiplies, and the number of live
// warps above which a launch uses them (kSoftPerSub per SM sub-partition).  A
// warp alone is limited by its chain of operations, where a software operation
// (~100 cycles) is slower than the unit's 64; from three warps per sub-partition
// on the unit and the integer pipes share the work.  Above two, three: 45,000
// rollouts 16.0, 21.4 ms (paper preset 20.6, 27.6; braking lead 14.1, 19.4);
// at 30,000 and from 65,000 on alike.  (A warp alone with only the position's last
// product and sum in software: 11.35 -> 11.5 ms at 1e4, so its chain is the limit,
// not the unit's rate.)
constexpr unsigned kSoftPerSub = 2;
struct SoftStep {
    SoftFactor h2, dt, h6;
    bool ok;
    unsigned above;
};

// Bounds of the states the fused forms are used on: they keep every sum and
// product of a step below 2^400, so nothing overflows.
constexpr int kTtcSpan = 256;  // steps one trigger test may cover
constexpr int kRunHeld = 64, kRunPiece = 16;  // steps of a run (a piece's end in a hold is seen after it)
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

// Realised deceleration r for demand D = -a (Eq. 5 as printed, or the per-axle
// fixed point min(min(D, mu gc), min(f0 + f1 D, r0 + r1 D)); c: the constant cap).
template <int CAP>
__device__ __forceinline__ double realised(double f0, double f1, double r0, double r1, double c,
                                           double D)
{
    if (CAP == AEB_CAP_LUMPED) return dmin(D, c);
    double lf = f0 + f1 * D;
    double lr = r0 + r1 * D;
    return dmin(dmin(D, c), dmin(lf, lr));
}

// A warp's shared memory: the prepared samples of (up to 32 of) its ticket, and
// each lane's rarely read values in a column of its own.
enum { S_V0, S_D0, S_GS, S_K, S_IT, S_KEY, S_NCOPY,  // KEY: perception-key row, as bits
       S_F0 = S_NCOPY, S_F1, S_R0, S_R1, S_MG, S_NOISE, S_THR, S_N };
enum { K_F0, K_F1, K_R0, K_R1, K_MG, K_NOISE, K_THR, K_N };  // S_F0 + K_*
enum { B_RUN = 1, B_LAGGED = 2, B_ORDERED = 4, B_DAMPED = 8, B_SOFT = 16 };
struct WarpMem {
    double rec[S_N][32];
    double cold[K_N][32];
    float line[5][32], cline[5][32];  // f0, f1, r0, r1, mg (or cap) in binary32
    uint32_t pos[32];
    int32_t delay[32], bits[32];
};

// The line of r(D) that is the strict minimum at D and the demand interval, as
// order keys, on which it stays so (piece -1: none can be named).
struct Piece {
    int piece;
    long long klo, khi;
};

// In binary64: the interval shrunk by a band of 1e-12 relative.
__device__ __noinline__ Piece select_exact(bool lumped, double f0, double f1, double r0,
                                           double r1, double c, double D)
{
    Piece p{-1, 0, 0};
    const double A[4] = {0.0, lumped ? c : f0, r0, c};
    const double S[4] = {1.0, lumped ? 0.0 : f1, r1, 0.0};
    const int nl = lumped ? 2 : 4;
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
        if (!(fabs(ds) >= 1e-6) || !(val[j] > val[cur])) return p;
        const double B = (A[j] - A[cur]) / ds;  // line j meets the current line
        const double band = 1e-12 * (1.0 + fabs(A[j]) + fabs(A[cur]) + fabs(B)) / fabs(ds);
        if (ds > 0.0) hi = fmin(hi, B - band);  // line j is below beyond B
        else lo = fmax(lo, B + band);
    }
    if (!(lo <= D && D <= hi)) return p;
    p.klo = okey(lo);
    p.khi = okey(hi);
    p.piece = (lumped && cur == 1) ? 3 : cur;
    return p;
}

// In binary32, for demands that are not close to a breakpoint (binary64
// divisions cost ~1000 cycles each): the same with a band of 1e-5 relative
// (all slopes at most 8, at least 1e-3 apart), far above the rounding of the
// lines and of their crossings, so the line is the strict minimum on the
// interval in binary64 too.
__device__ __forceinline__ Piece select_fast(bool lumped, const float (*ln)[32], int lane, float D)
{
    Piece p{-1, 0, 0};
    const float c = ln[4][lane];
    const float A[4] = {0.0f, lumped ? c : ln[0][lane], ln[2][lane], c};
    const float S[4] = {1.0f, lumped ? 0.0f : ln[1][lane], ln[3][lane], 0.0f};
    const int nl = lumped ? 2 : 4;
    float cv = D, cA = 0.0f, cS = 1.0f;
    int cur = 0;
#pragma unroll
    for (int j = 1; j < 4; ++j) {
        if (j >= nl) continue;
        const float vj = fmaf(S[j], D, A[j]);
        if (vj < cv) {
            cv = vj;
            cA = A[j];
            cS = S[j];
            cur = j;
        }
    }
    const float inf = __int_as_float(0x7f800000);
    float lo = -inf, hi = inf;
    bool ok = fabsf(cS) <= 8.0f && fabsf(cA) < 1e6f;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        if (j >= nl || j == cur) continue;
        const float ds = cS - S[j];
        ok = ok && fabsf(ds) >= 1e-3f && fabsf(S[j]) <= 8.0f && fabsf(A[j]) < 1e6f;
        const float B = __fdividef(A[j] - cA, ds);
        const float band = __fdividef(1e-5f * (1.0f + fabsf(A[j]) + fabsf(cA) + fabsf(B)), fabsf(ds));
        if (ds > 0.0f) hi = fminf(hi, B - band);
        else lo = fmaxf(lo, B + band);
    }
    const float slack = 1e-6f * (1.0f + fabsf(D));  // D's own rounding
    if (!ok || !(lo + slack <= D && D + slack <= hi)) return p;
    p.klo = okey((double)lo);
    p.khi = okey((double)hi);
    p.piece = (lumped && cur == 1) ? 3 : cur;
    return p;
}

// A step by the plain expressions of the definition, for states outside the
// range of the fused forms or without ordered stage demands.
struct Plain {
    double x, v, a;
};
template <int CAP>
__device__ __noinline__ Plain plain_step(double x, double v, double a, double u, double it,
                                         bool lagged, double k, double gs, double f0, double f1,
                                         double r0, double r1, double c, double dt, double h2,
                                         double h6)
{
    double a1, a2, a3, a4, ka1 = 0.0, ka2 = 0.0, ka3 = 0.0, ka4 = 0.0;
    if (lagged) {
        a1 = a;
        ka1 = (u - a1) * it;
        a2 = a + h2 * ka1;
        ka2 = (u - a2) * it;
        a3 = a + h2 * ka2;
        ka3 = (u - a3) * it;
        a4 = a + dt * ka3;
        ka4 = (u - a4) * it;
    } else {
        a1 = a2 = a3 = a4 = u;
    }
    auto accel = [&](double vv, double aa) {
        const double r = realised<CAP>(f0, f1, r0, r1, c, -aa);
        return ((-r) - (k * vv) * vv) - gs;
    };
    const double kv1 = accel(v, a1);
    const double v2 = v + h2 * kv1;
    const double kv2 = accel(v2, a2);
    const double v3 = v + h2 * kv2;
    const double kv3 = accel(v3, a3);
    const double v4 = v + dt * kv3;
    const double kv4 = accel(v4, a4);
    Plain p;
    p.x = x + h6 * (((v + 2.0 * v2) + 2.0 * v3) + v4);
    p.v = v + h6 * (((kv1 + 2.0 * kv2) + 2.0 * kv3) + kv4);
    p.a = lagged ? a + h6 * (((ka1 + 2.0 * ka2) + 2.0 * ka3) + ka4) : u;
    return p;
}

// A bool known when compiling, for a generic lambda.
template <bool B>
struct Constant {
    __device__ __forceinline__ constexpr operator bool() const { return B; }
};

template <int CAP, bool LEAD, bool TTC>
struct Lane64 {
    double x, v, a;
    double d0, gs, k, it;
    double c;                     // the constant cap: mu g cos(theta), or the Eq. 5 cap
    double mc;                    // -c (a negation is an operation of the binary64 unit)
    double npa, pb;               // current line: -r = npa + pb a (piece 1, 2)
    long long klo, khi;           // its demand interval [dlo, dhi] as order keys
    int32_t n, n_b, n_delay;
    uint32_t pos;
    int piece;                    // 0: D, 1, 2: an axle line, 3: the constant cap; -1: none
    bool trig, lagged, ordered;
    bool active;                  // the lane holds a rollout
    bool soft;                    // k and 1 / tau are factors of software multiplies
    bool damped;                  // dt / tau <= 1: the stage demands approach -a_cmd from below
    bool held;                    // r is the same at every stage until onset, or for good
    double nr;                    // -r while held
    int32_t n_chk;                // TTC: no step before this one can trigger
    WarpMem *mem;
    int lane;

    __device__ __forceinline__ double cold(int f) const { return mem->cold[f][lane]; }

    __device__ __forceinline__ void select_piece(double D)
    {
        piece = -1;
        if (!ordered) return;
        Piece p = select_fast(CAP == AEB_CAP_LUMPED, mem->cline, lane, (float)D);
        if (p.piece < 0)
            p = select_exact(CAP == AEB_CAP_LUMPED, cold(K_F0), cold(K_F1), cold(K_R0),
                             cold(K_R1), c, D);
        piece = p.piece;
        klo = p.klo;
        khi = p.khi;
        if (CAP != AEB_CAP_LUMPED && piece >= 0) {
            npa = -cold(piece == 2 ? K_R0 : K_F0);
            pb = cold(piece == 2 ? K_R1 : K_F1);
        }
    }

    // dv/dt from -r: (-r - (k v) v) - g sin(theta).
    __device__ __forceinline__ double accel(const Ops &q, double vv, double mr) const
    {
        return q.sub(q.sub(mr, q.mul(q.mul(k, vv), vv)), gs);
    }
    // The same with the products on the integer pipes.
    __device__ __forceinline__ double accel_soft(const Ops &q, const SoftFactor &fk, double vv,
                                                 double mr, uint32_t &range) const
    {
        const double t = soft_mul(soft_mul(vv, fk, range), soft_factor(vv), range);
        return q.sub(q.sub(mr, t), gs);
    }
    // -r on the current piece (or held): the same value as the full minimum's
    // for a demand -aa in the piece's interval (pa + pb (-aa) and npa + pb aa
    // round alike).  `lines`: some lane of the warp
    // is on an axle line.
    __device__ __forceinline__ double r_piece(const Ops &q, double aa, bool lines) const
    {
        double mr = (piece == 0) ? aa : mc;
        if (CAP != AEB_CAP_LUMPED && lines) {
            const double rl = q.add(npa, q.mul(pb, aa));
            if (piece == 1 || piece == 2) mr = rl;
        }
        return held ? nr : mr;
    }
    __device__ __forceinline__ double r_piece_soft(const Ops &q, const SoftFactor &fb, double aa,
                                                   bool lines, uint32_t &range) const
    {
        double mr = (piece == 0) ? aa : mc;
        if (CAP != AEB_CAP_LUMPED && lines) {
            uint32_t rg = 0;
            const double rl = q.add(npa, soft_mul(aa, fb, rg));
            if (piece == 1 || piece == 2) {
                mr = rl;
                if (!held) range |= rg;
            }
        }
        return held ? nr : mr;
    }
    // -r by the full minimum in fused forms (finite lines; order keys compare
    // as the values).
    __device__ __forceinline__ double r_full(const Ops &q, double aa) const
    {
        auto kmin = [](double a, double b) { return okey(b) < okey(a) ? b : a; };
        const double D = -aa;
        if (CAP == AEB_CAP_LUMPED) return held ? nr : -kmin(D, c);
        const double lf = q.add(cold(K_F0), q.mul(cold(K_F1), D));
        const double lr = q.add(cold(K_R0), q.mul(cold(K_R1), D));
        return held ? nr : -kmin(kmin(D, c), kmin(lf, lr));
    }

    // Hold r at the actuator value aa, at which the lane stays until onset (0)
    // or for good (an instantaneous or settled actuator's command).
    __device__ __forceinline__ void hold_at(double aa)
    {
        held = ordered;
        nr = -realised<CAP>(cold(K_F0), cold(K_F1), cold(K_R0), cold(K_R1), c, -aa);
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
            nr = mc;
        } else if (__double_as_longlong(a) == __double_as_longlong(M.a_cmd)) {
            hold_at(a);  // settled: a does not move any more
        }
    }

    // Whether k is negative (of the model's constants only finiteness is asked:
    // an air density or area may be): then the car's speed has no bound over a
    // span of steps, so that every step tests the trigger and a moving lead.
    __device__ __forceinline__ bool driven() const { return __double2hiint(k) < 0; }

    __device__ __forceinline__ int32_t onset() const
    {
        return TTC ? (trig ? n_b : -1) : n_delay;
    }

    // Take the prepared sample `slot`.
    __device__ __forceinline__ void take(int slot)
    {
        const WarpMem &w = *mem;
        v = w.rec[S_V0][slot];
        d0 = w.rec[S_D0][slot];
        gs = w.rec[S_GS][slot];
        k = w.rec[S_K][slot];
        it = w.rec[S_IT][slot];
        c = w.rec[S_MG][slot];
        mc = -c;
#pragma unroll
        for (int f = 0; f < K_N; ++f) mem->cold[f][lane] = w.rec[S_F0 + f][slot];
#pragma unroll
        for (int f = 0; f < 5; ++f) mem->cline[f][lane] = w.line[f][slot];
        if (TTC) mem->cold[K_MG][lane] = w.rec[S_KEY][slot];  // (c is in a register)
        pos = w.pos[slot];
        n_delay = w.delay[slot];
        const int b = w.bits[slot];
        lagged = b & B_LAGGED;
        ordered = b & B_ORDERED;
        damped = b & B_DAMPED;
        soft = b & B_SOFT;
        trig = !TTC;
        n_b = n_delay;
        x = 0.0;
        a = 0.0;
        n = 0;
        n_chk = 0;
        select_piece(-a);
        hold_at(a);
    }

    // TTC trigger (while not yet triggered), at the start of step n.  A test
    // that does not fire also bounds the steps that cannot (n_chk): while r is
    // held the car's acceleration is at most acc = max(0, -r - g sin(theta)),
    // so over kTtcSpan steps its speed stays below W = v + kTtcSpan dt acc and
    // the margin (gap + noise) - thr c falls by at most dt (W + |thr| rate) per
    // step (a braking lead's travel only widens the gap).  rate bounds the
    // closing speed's change towards the trigger: for thr >= 0 its rise, acc and
    // the lead's b_L; for thr < 0 its fall, r + g sin(theta) and the drag at W,
    // as long as one step of that keeps every stage speed within [-W, W].  A
    // reading's noise is at most 3 perc_sigma.  (None of this holds for a drag
    // that drives the car, see driven().)
    __device__ __forceinline__ void test_trigger(const ModelDev &M, const Ops &q)
    {
        double gap_meas, closing;
        if (M.lead_moving) {  // gap and closing speed to the moving lead
            const double t = from_int(n) * q.dt;
            gap_meas = ((d0 + lead_pos(M, t)) - x) + cold(K_NOISE);
            closing = v - lead_speed(M, t);
        } else {
            gap_meas = q.add(q.sub(d0, x), cold(K_NOISE));
            closing = v;
        }
        const double thr = cold(K_THR);
        const double limit = q.mul(thr, closing);
        const float margin = (float)(gap_meas - limit) - 3.001f * (float)M.perc_sigma;
        bool reading = true;
        if (M.perc && !(margin > 0.0f)) {  // the reading of step n + L describes step n
            uint32_t h[4];
            perc_halves((uint64_t)__double_as_longlong(cold(K_MG)), (uint64_t)((long long)n + M.perc_lat), M.perc_seed, h);
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
        } else if (held && margin > 0.0f && tame_speed(v) && !driven()) {
            const float dtf = (float)q.dt, net = (float)(nr - gs), acc = fmaxf(0.0f, net);
            const float W = (float)v + (float)kTtcSpan * dtf * acc;
            const bool rising = __double2hiint(thr) >= 0;  // (the sign: -0 has no term)
            const float rate = rising ? acc + (float)M.lead_decel
                                      : fmaxf(0.0f, -net) + (float)k * W * W;
            const float fall = dtf * (W + fabsf((float)thr) * rate) * 1.001f;
            // margin's own rounding: a few binary32 ulps of what it was formed from
            const float m = margin * 0.999f - 1e-5f * (fabsf((float)gap_meas) + fabsf((float)limit));
            const float steps = __fdividef(m, fall);
            if (steps > 1.0f && (rising || dtf * rate * 1.001f <= W))
                n_chk = n + (steps < (float)kTtcSpan ? (int)steps : kTtcSpan);
        }
    }

    // The end of the step from (x0, v0) at step n0 to (x1, v1): contact, stop or
    // the horizon, refined and stored; false if the rollout goes on.
    __device__ __forceinline__ bool finish(const ModelDev &M, const Ops &q, const OutDev &O,
                                           const WorkDev &W, double x0, double v0, int32_t n0,
                                           double x1, double v1) const
    {
        const double dt = q.dt;
        if (LEAD && M.lead_moving) {
            const double t0 = from_int(n0) * dt, t1 = from_int(n0 + 1) * dt;
            const double g1 = (d0 + lead_pos(M, t1)) - x1;
            if (g1 <= 0.0) {
                const double g0 = (d0 + lead_pos(M, t0)) - x0;
                const double c0 = v0 - lead_speed(M, t0), c1 = v1 - lead_speed(M, t1);
                const double s = g0 / (g0 - g1);
                store_out(O, row_of(W, pos, 0.0).o, AEB_CONTACT, x1, x0 + s * (x1 - x0),
                          c0 + s * (c1 - c0), ((double)n0 + s) * dt, n0 + 1, onset());
                return true;
            }
        } else if (LEAD && ge_pos(x1, d0)) {  // d0 > 0 and finite here
            const double s = (d0 - x0) / (x1 - x0);
            store_out(O, row_of(W, pos, 0.0).o, AEB_CONTACT, x1, d0, v0 + s * (v1 - v0),
                      ((double)n0 + s) * dt, n0 + 1, onset());
            return true;
        }
        if (le_zero(v1)) {
            const double s = v0 / (v0 - v1);
            store_out(O, row_of(W, pos, 0.0).o, AEB_STOP, x1, x0 + s * (x1 - x0), 0.0,
                      ((double)n0 + s) * dt, n0 + 1, onset());
            return true;
        }
        if (n0 + 1 >= M.n_max) {
            store_out(O, row_of(W, pos, 0.0).o, AEB_HORIZON, x1, x1, 0.0, (double)(n0 + 1) * dt,
                      n0 + 1, onset());
            return true;
        }
        return false;
    }

    // How many steps from here need none of step()'s event tests: before the
    // horizon's last step, the onset, the next trigger test and, with a moving
    // lead, before the gap can have closed (the car's acceleration is at most
    // |g sin(theta)| while its demand is not negative; the lead's travel only
    // widens the gap).
    __device__ __forceinline__ int room(const ModelDev &M, const Ops &q) const
    {
        if (!active) return kRunHeld;
        if (!(ordered && tame_speed(v) && (held || piece >= 0))) return 0;
        int r = min(kRunHeld, (M.n_max - 1) - n);
        if (TTC && !trig) r = min(r, n_chk - n);
        else if (n <= n_b) r = min(r, n_b - n);
        if (LEAD && M.lead_moving && r > 0) {
            if (!(a <= 0.0 && c >= 0.0 && M.a_cmd <= 0.0 && !driven() &&
                  (held ? nr <= 0.0
                        : piece == 0 || piece == 3 || (npa <= 0.0 && pb >= 0.0))))
                return 0;
            const double xl = lead_pos(M, from_int(n) * q.dt);
            const float g = (float)((d0 + xl) - x) * 0.999f -
                            1e-5f * (fabsf((float)d0) + fabsf((float)xl) + fabsf((float)x));
            const float dtf = (float)q.dt;
            const float W = (float)v + (float)kRunHeld * dtf * fabsf((float)gs);
            const float steps = __fdividef(g, W * dtf * 1.001f);
            r = steps >= (float)r ? r : steps > 0.0f ? (int)steps : 0;
        }
        return r;
    }

    // One step with r held, from (x, v).
    template <bool SOFT>
    __device__ __forceinline__ void held_step(const Ops &q, const SoftStep &S, const SoftFactor &fk,
                                              double &xn, double &vn, uint32_t &rg) const
    {
        if (SOFT) {
            double vj = v, kj = accel_soft(q, fk, v, nr, rg), sv = v, sk = kj;
#pragma unroll 1
            for (int st = 0; st < 3; ++st) {  // (a loop: the instruction caches bound this)
                const SoftFactor fs = st < 2 ? S.h2 : S.dt;
                const double w = st < 2 ? q.two : q.one;
                vj = soft_add<false>(v, soft_mul(kj, fs, rg), rg);
                kj = accel_soft(q, fk, vj, nr, rg);
                sv = __fma_rn(w, vj, sv);
                sk = __fma_rn(w, kj, sk);
            }
            xn = soft_add<false>(x, soft_mul(sv, S.h6, rg), rg);
            vn = soft_add<false>(v, soft_mul(sk, S.h6, rg), rg);
        } else {
            const double kv1 = accel(q, v, nr);
            const double v2 = q.add(v, q.mul(q.h2, kv1));
            const double kv2 = accel(q, v2, nr);
            const double v3 = q.add(v, q.mul(q.h2, kv2));
            const double kv3 = accel(q, v3, nr);
            const double v4 = q.add(v, q.mul(q.dt, kv3));
            const double kv4 = accel(q, v4, nr);
            xn = q.combine(x, v, v2, v3, v4);
            vn = q.combine(v, kv1, kv2, kv3, kv4);
        }
    }

    // One step inside a piece (or held), from (x, v, a); `in`: the stage demands
    // lie in the piece's interval.  With dt / tau <= 2 they lie between the first
    // and the fourth (-a1 smallest when the command is a deceleration, so that
    // a - u >= 0 from the start, -a4 smallest otherwise): two tests for the step.
    // (The lag is stable and the stage actuator values are finite, so order keys
    // compare them.)  A lane that is not held has a lag.
    template <bool SOFT>
    __device__ __forceinline__ void piece_step(const ModelDev &M, const Ops &q, const SoftStep &S,
                                               const SoftFactor &fk, double u, bool lines,
                                               double &xn, double &vn, double &an, bool &in,
                                               uint32_t &rg) const
    {
        const bool dec = M.a_cmd <= 0.0;
        if (SOFT) {
            // (a held lane's actuator is not read: stand-ins keep it in range)
            const SoftFactor fi = soft_factor(it), fb = soft_factor(pb);
            const double a1 = held ? -1.0 : a, us = held ? -3.0 : u;
            uint32_t ra = lines && !held && !soft_factor_ok(pb) ? ~0u : 0u;
            double vj = v, aj = a1, kj = 0.0, kaj = 0.0, sv = v, sk = 0.0, sa = 0.0;
#pragma unroll 1
            for (int st = 0; st < 4; ++st) {
                if (st > 0) {
                    const SoftFactor fs = st < 3 ? S.h2 : S.dt;
                    aj = soft_add<true>(a1, soft_mul(kaj, fs, ra), ra);
                    vj = soft_add<false>(v, soft_mul(kj, fs, rg), rg);
                }
                kaj = soft_mul(q.sub(us, aj), fi, ra);
                kj = accel_soft(q, fk, vj, r_piece_soft(q, fb, aj, lines, rg), rg);
                if (st > 0) {
                    const double w = st < 3 ? q.two : q.one;
                    sv = __fma_rn(w, vj, sv);
                    sk = __fma_rn(w, kj, sk);
                    sa = __fma_rn(w, kaj, sa);
                } else {
                    sk = kj;
                    sa = kaj;
                }
            }
            an = soft_add<true>(a1, soft_mul(sa, S.h6, ra), ra);
            xn = soft_add<false>(x, soft_mul(sv, S.h6, rg), rg);
            vn = soft_add<false>(v, soft_mul(sk, S.h6, rg), rg);
            const long long kfirst = -okey(dec ? a1 : aj), klast = -okey(dec ? aj : a1);
            in = held || (kfirst >= klo && klast <= khi && !soft_bad(ra));
        } else {
            const double ka1 = q.mul(q.sub(u, a), it);
            const double a2 = q.add(a, q.mul(q.h2, ka1));
            const double ka2 = q.mul(q.sub(u, a2), it);
            const double a3 = q.add(a, q.mul(q.h2, ka2));
            const double ka3 = q.mul(q.sub(u, a3), it);
            const double a4 = q.add(a, q.mul(q.dt, ka3));
            const double ka4 = q.mul(q.sub(u, a4), it);
            const double kv1 = accel(q, v, r_piece(q, a, lines));
            const double v2 = q.add(v, q.mul(q.h2, kv1));
            const double kv2 = accel(q, v2, r_piece(q, a2, lines));
            const double v3 = q.add(v, q.mul(q.h2, kv2));
            const double kv3 = accel(q, v3, r_piece(q, a3, lines));
            const double v4 = q.add(v, q.mul(q.dt, kv3));
            const double kv4 = accel(q, v4, r_piece(q, a4, lines));
            an = q.combine(a, ka1, ka2, ka3, ka4);
            xn = q.combine(x, v, v2, v3, v4);
            vn = q.combine(v, kv1, kv2, kv3, kv4);
            const long long kfirst = -okey(dec ? a : a4), klast = -okey(dec ? a4 : a);
            in = held || (kfirst >= klo && klast <= khi);
        }
    }

    // Up to R (>= 1, warp-uniform, within room() of every lane) steps with no
    // event among them; true if the lane's rollout ended (stored).  The state a
    // step starts from is tested while the step is computed, and a step that
    // turns out not to exist (a lane had ended) or not to stay in a piece is
    // dropped: the tests' ~100 dependent integer instructions, which a warp
    // alone on its sub-partition would wait for, run beside the binary64 unit.
    // `redo`: the next step is one for step().
    template <bool SOFT>
    __device__ __forceinline__ bool run(const ModelDev &M, const Ops &q, const SoftStep &S,
                                        const OutDev &O, const WorkDev &W, int R, bool &redo)
    {
        const bool braking = trig && n >= n_b;
        const double u = braking ? M.a_cmd : 0.0;
        const SoftFactor fk = soft_factor(k);
        double x0 = x, v0 = v;  // the last step's start
        bool e = false;         // (x, v) ends the rollout, or leaves the range of the fused forms
        int done = 0;
        redo = false;
        auto advance = [&](double xn, double vn) {
            x0 = x;
            v0 = v;
            x = xn;
            v = vn;
            ++done;
            e = active && (!tame_speed(v) || le_zero(v) || (LEAD && !M.lead_moving && ge_pos(x, d0)));
        };
        if (__all_sync(kFull, !active || held)) {
#pragma unroll 1
            do {
                double xn, vn;
                uint32_t rg = 0;
                held_step<SOFT>(q, S, fk, xn, vn, rg);
                if (__any_sync(kFull, e)) break;
                if (SOFT && __any_sync(kFull, active && soft_bad(rg))) {
                    redo = true;
                    break;
                }
                advance(xn, vn);
            } while (done < R);
        } else {
            R = min(R, kRunPiece);
            // (on the unit a loop each for warps with and without a lane on an
            // axle line: a test inside the step cuts it into short blocks, 4480
            // against 3850 cycles for a warp alone; with software arithmetic one
            // loop: two wait on the instruction caches, 186 against 169 ms per 1e6)
            auto loop = [&](auto lines) {
#pragma unroll 1
                do {
                    double xn, vn, an;
                    bool in;
                    uint32_t rg = 0;
                    piece_step<SOFT>(M, q, S, fk, u, lines, xn, vn, an, in, rg);
                    if (__any_sync(kFull, e)) break;
                    if (!__all_sync(kFull, !active || (in && !(SOFT && soft_bad(rg))))) {
                        redo = true;
                        break;
                    }
                    if (!held) a = an;
                    advance(xn, vn);
                } while (done < R);
            };
            const bool lines = CAP != AEB_CAP_LUMPED &&
                               __any_sync(kFull, active && !held && (piece == 1 || piece == 2));
            if (SOFT) loop(lines);
            else if (lines) loop(Constant<true>{});
            else loop(Constant<false>{});
        }
        if (!active) return false;
        n += done;
        if (e && finish(M, q, O, W, x0, v0, n - 1, x, v)) return true;
        if (braking && !held && done > 0) try_hold(M);
        return false;
    }

    // One RK4 step with every event it may meet, on the binary64 unit (all lanes
    // of the warp together); true if the lane's rollout ended (stored).
    __device__ __forceinline__ bool step(const ModelDev &M, const Ops &q, const OutDev &O,
                                         const WorkDev &W)
    {
        const double dt = q.dt, h2 = q.h2, h6 = q.h6;
        if (TTC && active && !trig && n >= n_chk) test_trigger(M, q);
        if (trig && n == n_b) {  // the command switches on: a moves from here, or has moved
            held = false;
            if (!lagged) hold_at(M.a_cmd);
        }
        const bool braking = trig && n >= n_b;
        const double u = braking ? M.a_cmd : 0.0;
        const bool fused = ordered && tame_speed(v);
        double v2, v3, v4, xn, vn, an;
        bool pw = true;
        if (__all_sync(kFull, !active || (held && fused))) {
            const double kv1 = accel(q, v, nr);
            v2 = q.add(v, q.mul(h2, kv1));
            const double kv2 = accel(q, v2, nr);
            v3 = q.add(v, q.mul(h2, kv2));
            const double kv3 = accel(q, v3, nr);
            v4 = q.add(v, q.mul(dt, kv3));
            const double kv4 = accel(q, v4, nr);
            xn = q.combine(x, v, v2, v3, v4);
            vn = q.combine(v, kv1, kv2, kv3, kv4);
            an = lagged ? a : u;  // not read while r is held
        } else {
            if (__any_sync(kFull, active && fused)) {
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
                // (the stage demands in order, as in piece_step)
                const bool dec = M.a_cmd <= 0.0;
                const long long kfirst = -okey(dec ? a1 : a4), klast = -okey(dec ? a4 : a1);
                pw = held || (piece >= 0 && kfirst >= klo && klast <= khi);
                double kv1, kv2, kv3, kv4;
                if (__all_sync(kFull, !active || !fused || pw)) {
                    const bool lines =
                        __any_sync(kFull, active && !held && (piece == 1 || piece == 2));
                    kv1 = accel(q, v, r_piece(q, a1, lines));
                    v2 = q.add(v, q.mul(h2, kv1));
                    kv2 = accel(q, v2, r_piece(q, a2, lines));
                    v3 = q.add(v, q.mul(h2, kv2));
                    kv3 = accel(q, v3, r_piece(q, a3, lines));
                    v4 = q.add(v, q.mul(dt, kv3));
                    kv4 = accel(q, v4, r_piece(q, a4, lines));
                } else {
                    // some lane crosses a breakpoint: the full minimum for the
                    // warp (67 operations, where the lane alone would add them
                    // to the others' 51-59)
                    kv1 = accel(q, v, r_full(q, a1));
                    v2 = q.add(v, q.mul(h2, kv1));
                    kv2 = accel(q, v2, r_full(q, a2));
                    v3 = q.add(v, q.mul(h2, kv2));
                    kv3 = accel(q, v3, r_full(q, a3));
                    v4 = q.add(v, q.mul(dt, kv3));
                    kv4 = accel(q, v4, r_full(q, a4));
                }
                xn = q.combine(x, v, v2, v3, v4);
                vn = q.combine(v, kv1, kv2, kv3, kv4);
                an = lagged ? q.combine(a, ka1, ka2, ka3, ka4) : u;
                if (held && lagged) an = a;
            }
            if (active && !fused) {
                const Plain p = plain_step<CAP>(x, v, a, u, it, lagged, k, gs, cold(K_F0),
                                                cold(K_F1), cold(K_R0), cold(K_R1), c, dt, h2, h6);
                xn = p.x;
                vn = p.v;
                an = p.a;
                pw = false;
            }
        }
        if (!active) return false;
        if (finish(M, q, O, W, x, v, n, xn, vn)) return true;
        x = xn;
        v = vn;
        a = an;
        n = n + 1;
        if (!pw) select_piece(-a);
        else if (braking && !held) try_hold(M);
        return false;
    }
};

// Prepare entries [start, start + cnt) of the processing order (cnt <= 32) into
// the warp's records, one per lane: the set-up's binary64 divisions run once per
// ticket at full width instead of once per refilling lane.  Samples that end at
// once are stored here.
template <int CAP, bool LEAD, bool TTC>
__device__ __noinline__ void prepare(const ModelDev &M, const ParamsDev &P, const OutDev &O,
                                     const WorkDev &W, uint32_t start, int cnt, WarpMem &w)
{
    const int j = threadIdx.x & 31;
    if (j >= cnt) return;
    const uint32_t pos = position(W, start + (uint32_t)j);
    const Row rows = row_of(W, pos, M.ttc_thr);
    const uint64_t i = rows.o;
    double f[AEB_NFIELDS];
    load_fields(P, rows.p, f);
    w.bits[j] = 0;
    if (!sample_valid(f)) {
        const double nan = __longlong_as_double(0x7ff8000000000000ll);
        store_out(O, i, AEB_INVALID, nan, nan, nan, nan, 0, -1);
        return;
    }
    const double k = ((M.rho * f[kCd]) * M.area) / (2.0 * f[kMass]);
    const bool lagged = f[kTau] > 0.0;
    const double it = lagged ? 1.0 / f[kTau] : 0.0;
    const double mu = f[kMu], mh = mu * M.hl;
    double c, f0 = 0.0, f1 = 0.0, r0 = 0.0, r1 = 0.0;
    if (CAP == AEB_CAP_LUMPED) {
        c = (mu * M.g) / (1.0 + mh);
    } else {
        c = mu * f[kGc];
        f0 = (c * M.phi_f) / (1.0 - mh);
        f1 = (1.0 - M.beta) / (1.0 - mh);
        r0 = (c * (1.0 - M.phi_f)) / (1.0 + mh);
        r1 = M.beta / (1.0 + mh);
    }
    const int32_t n_delay = steps_to_reach_dev(f[kTdelay], M.dt);
    const int32_t on = TTC ? -1 : n_delay;
    if (LEAD && f[kD0] <= 0.0) {
        store_out(O, i, AEB_CONTACT, 0.0, 0.0, f[kV0], 0.0, 0, on);
        return;
    }
    if (f[kV0] <= 0.0) {
        store_out(O, i, AEB_STOP, 0.0, 0.0, 0.0, 0.0, 0, on);
        return;
    }
    if (M.n_max == 0) {
        store_out(O, i, AEB_HORIZON, 0.0, 0.0, 0.0, 0.0, 0, on);
        return;
    }
    // ordered: stage demands in order, and the sample inside the range of the
    // fused forms (see Ops)
    const bool ordered = (!lagged || M.dt * it <= 2.0) && M.dt >= 1e-30 && M.dt <= 1.0 &&
                         fabs(M.a_cmd) <= kTame && k <= 1.0 && fabs(f[kGs]) <= kTame &&
                         fabs(c) < 1e50 && fabs(f0) < 1e50 && fabs(f1) < 1e50 &&
                         fabs(r0) < 1e50 && fabs(r1) < 1e50;
    const bool damped = lagged && M.dt * it <= 1.0 && M.a_cmd < 0.0;
    w.rec[S_V0][j] = f[kV0];
    w.rec[S_D0][j] = f[kD0];
    w.rec[S_GS][j] = f[kGs];
    w.rec[S_K][j] = k;
    w.rec[S_IT][j] = it;
    w.rec[S_KEY][j] = __longlong_as_double((long long)rows.k);
    w.rec[S_F0][j] = f0;
    w.rec[S_F1][j] = f1;
    w.rec[S_R0][j] = r0;
    w.rec[S_R1][j] = r1;
    w.rec[S_MG][j] = c;
    w.rec[S_NOISE][j] = f[kNoise];
    w.rec[S_THR][j] = rows.thr;
    w.line[0][j] = (float)f0;
    w.line[1][j] = (float)f1;
    w.line[2][j] = (float)r0;
    w.line[3][j] = (float)r1;
    w.line[4][j] = (float)c;
    w.pos[j] = pos;
    w.delay[j] = n_delay;
    w.bits[j] = B_RUN | (lagged ? B_LAGGED : 0) | (ordered ? B_ORDERED : 0) |
                (damped ? B_DAMPED : 0) |
                (soft_factor_ok(k) && (!lagged || soft_factor_ok(it)) ? B_SOFT : 0);
}

#ifndef AEB_FP64_MIN_BLOCKS
#define AEB_FP64_MIN_BLOCKS 4  // resident blocks per SM the register budget must allow
#endif

template <int CAP, bool LEAD, bool TTC>
__global__ void __launch_bounds__(128, AEB_FP64_MIN_BLOCKS)
k_rollout_fp64(ModelDev M, SoftStep S, ParamsDev P, OutDev O, WorkDev W)
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
    __shared__ WarpMem mem[4];
    WarpMem &w = mem[threadIdx.x >> 5];
    Ticket ticket{0, 0, false};
    int batched = 0;         // entries of the ticket already prepared
    int used = 0, cnt = 0;   // prepared samples taken, and how many there are
    bool dry = false;
    Lane64<CAP, LEAD, TTC> L;
    L.mem = &w;
    L.lane = (int)lane;
    L.active = false;
    L.x = L.v = L.a = L.d0 = L.gs = L.k = L.it = L.c = L.mc = L.npa = L.pb = L.nr = 0.0;
    L.klo = L.khi = 0;
    L.n = L.n_b = L.n_delay = L.n_chk = 0;
    L.pos = 0;
    L.piece = -1;
    L.trig = L.lagged = L.ordered = L.damped = L.held = L.soft = false;
    // Software arithmetic pays while the sub-partitions hold enough warps
    // (see SoftStep): decided from the launch, and again, once the tickets are
    // out, from the warps that have ended.  Both ways give the same bits.
    unsigned long long *ended = W.counter + 1;
    const unsigned warps = gridDim.x * 4u;
    bool use_soft = warps > S.above;
    unsigned runs = 0;
    unsigned need = kFull;
    for (;;) {
        while (need) {
            if (used >= cnt) {
                if (!dry && batched >= ticket.count) {
                    ticket = claim_ticket(W);
                    batched = 0;
                    dry = !ticket.ok;
                }
                if (dry) {
                    if ((need >> lane) & 1u) L.active = false;
                    break;
                }
                cnt = min(32, ticket.count - batched);
                used = 0;
                __syncwarp();  // every lane has read its record of the previous batch
                prepare<CAP, LEAD, TTC>(M, P, O, W, ticket.start + (uint32_t)batched, cnt, w);
                __syncwarp();
                batched += cnt;
            }
            const int slot = used + __popc(need & lanemask_lt());
            const bool got = ((need >> lane) & 1u) && slot < cnt;
            if (got) {
                L.active = w.bits[slot] & B_RUN;
                if (L.active) L.take(slot);
            }
            const unsigned taken = __ballot_sync(kFull, got);
            used += __popc(taken);
            // (a sample that ended at once leaves its lane in need)
            need = (need & ~taken) | __ballot_sync(kFull, got && !L.active);
        }
        if (!__any_sync(kFull, L.active)) {
            if (lane == 0) atomicAdd(ended, 1ull);
            return;
        }
        const int R = __reduce_min_sync(kFull, L.room(M, q));
        need = 0;
        bool redo = true;
        if (R > 0) {
            if (use_soft && dry && (++runs & 3u) == 0u) {
                // (one reading for the warp: the lanes must agree on the way they
                // take, which has full-warp votes of its own)
                unsigned gone = 0;
                if (lane == 0) gone = (unsigned)*(volatile unsigned long long *)ended;
                use_soft = warps - __shfl_sync(kFull, gone, 0) > S.above;
            }
            const bool soft = use_soft && S.ok && __all_sync(kFull, !L.active || L.soft);
            const bool over = soft ? L.template run<true>(M, q, S, O, W, R, redo)
                                   : L.template run<false>(M, q, S, O, W, R, redo);
            need = __ballot_sync(kFull, over);
        }
        if (redo) need = __ballot_sync(kFull, L.step(M, q, O, W));
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
    const SoftStep st{soft_factor(m.h2), soft_factor(m.dt), soft_factor(m.h6),
                      soft_factor_ok(m.h2) && soft_factor_ok(m.dt) && soft_factor_ok(m.h6),
                      kSoftPerSub * 4u * (unsigned)sms};
    kern<<<(unsigned)blocks, 128, 0, s>>>(m, st, p, o, w);
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
