// mlkd_pair.cuh -- one correlated fine/coarse pair as a register-resident
// state machine, shared by the per-level kernel and the batched kernel.
//
//   pair_start : Alg. 1 / Alg. 2 initialisation (nu_0, E_0 shared by both
//                paths, x_0).
//   pair_event : one fine KD event (Alg. 1 KineticDiffusionStep) and, when
//                the new fine collision lies at or after the end of the
//                current coarse step, the coarse KD step built from the
//                aggregated random numbers (Sec. 3.1 mapping, Sec. 3.2
//                aggregation, Alg. 2).
//   pair_drift : the final kinetic move of both paths to T.
// Time is an integer count of fine steps plus a flight in fine-step units,
// so the coarse collision equals the fine collision kappa_k exactly.
#pragma once

#include <type_traits>

#include "mlkd_internal.h"

namespace mlkd {

// Observer of the coarse steps (validation only): pair_event calls
// tr->coarse(nu~, E~, chi~) at each coarse KD step when a tracer is given.
// NoTrace compiles to nothing.
struct NoTrace {};

// FP64 state is dimensionless: with velocities mu + sigma nu, the position
// is x = x_0 + mu t + (sigma/R) y, a kinetic phase of optical length E moves y by
// nu E, and no coefficient of the background is left in the KD step but R dt.
// xf, xc hold y and vf, vc hold nu.  A flight is kept as its optical length and
// its split into whole steps and the rest of the collision's step.
// FP32 keeps the flight in fine steps and its floor.
template <typename Real> struct FlightState {
    Real qf, qc;
    int whole_f;                // floor(qf)
};
template <> struct FlightState<double> {
    double x0;                  // initial position
    double of, oc;              // optical lengths E of the fine and coarse flights
    uint64_t left_f, left_c;    // 2^64 (whole + 1 - flight in steps)
    int whole_f, whole_c;
};

template <typename Real> struct PairState : FlightState<Real> {
    Real xf, vf;                // fine path: position, velocity
    Real xc, vc;                // coarse path
    Real num, den, chi_first;   // streamed eq. chi-update of the open coarse window
    int i_f, ic, Ec;            // fine-step index of each path's phase start; coarse step end
    uint32_t k, evc;            // fine events (= Philox block of the next draw - 1), coarse events
    uint32_t pair_lo, word2;    // Philox counter words of this pair
    bool fresh;                 // the open window has no term yet
};

template <typename Real> struct LevelCtx {
    Background<Real> bg;
    int n;                      // fine steps to T on this level
    int M;                      // refinement factor
    DivM divM;                  // floor(n / M)
    int init;                   // 0: x0 = 0; 1: cosine density
    uint32_t word2;             // level << 24
    uint32_t request;
};

// End of the coarse step that contains fine-step position base + steps + f
// (0 <= f < 1), with base on the coarse grid: base + M (steps / M + 1).
template <typename Real>
__device__ __forceinline__ int next_coarse_end(const LevelCtx<Real> &L, int base, int steps)
{
    return base + L.M * (L.divM(steps) + 1);
}

// CPL: 0 = level 0 (single path), 1 = coupled pair, 2 = decided at run time.
template <typename Real, int CPL>
__device__ __forceinline__ bool pair_is_coupled(bool runtime) { return CPL == 2 ? runtime : CPL == 1; }

// Position x at T from the FP64 pair state.  c = sigma/R enters as the sum of
// two numbers: rounded to one it would shift every pair's x alike.
__device__ __forceinline__ double position_at_T(const LevelCtx<double> &L, double x0, double y)
{
    return fma(L.bg.c, y, fma(L.bg.c_lo, y, fma(L.bg.mu, (double)L.n * L.bg.dt, x0)));
}

// A pair's first flight, drawn as E (FP64) or in fine steps (FP32): in fine
// steps, and whether its collision lies before T.
template <typename Real> __device__ __forceinline__ Real first_flight(const LevelCtx<Real> &L, Real q0)
{
    if constexpr (std::is_same<Real, double>::value) return q0 * L.bg.inv_Rdt;
    else return q0;
}
template <typename Real> __device__ __forceinline__ bool collides_before_T(const LevelCtx<Real> &L, Real q0)
{
    if constexpr (std::is_same<Real, double>::value)
        return fx::split_flight(fx::pos_of(first_flight(L, q0))).whole < L.n;
    else
        return q0 < (Real)L.n;
}

// Alg. 1 / Alg. 2 initialisation values of pair p: x_0, v_0 and the first
// flight (nu_0, E_0 and the initial-position uniform of Philox block 0),
// shared by both paths; FP64: nu_0 and E_0.
template <typename Real, int RECIPE = 0>
__device__ __forceinline__ void pair_start_values(Real &x0, Real &v0, Real &q0, unsigned long long p,
                                                  const LevelCtx<Real> &L, const PhiloxKeys &keys)
{
    if constexpr (std::is_same<Real, double>::value) {
        const DrawFixed d0 = draw_fixed_r<RECIPE>(0u, (uint32_t)p, L.word2 ^ (uint32_t)(p >> 32), L.request, keys);
        x0 = L.init ? cosine_inverse_fp64<RECIPE == 1 ? 24 : 53>(d0.n4) : 0.0;
        v0 = d0.nu_();
        q0 = fx::to_double(d0.E);
    } else {
        const Draw<Real> d0 = draw_r<Real, RECIPE>(0u, (uint32_t)p, L.word2 ^ (uint32_t)(p >> 32),
                                                   L.request, keys);
        x0 = L.init ? cosine_inverse<Real>(d0.u4) : Real(0);
        v0 = L.bg.mu + L.bg.sigma * d0.nu;
        q0 = d0.E * L.bg.inv_Rdt;
    }
}

// Both paths of the pair start at x0.
template <typename Real> __device__ __forceinline__ void set_start(PairState<Real> &st, Real x0)
{
    if constexpr (std::is_same<Real, double>::value) {
        st.x0 = x0;
        st.xf = st.xc = 0.0;
    } else {
        st.xf = st.xc = x0;
    }
}

// The state of pair p at t = 0 from its initialisation values.  Returns true
// if the pair has no collision before T (already finished).
template <typename Real, int CPL>
__device__ __forceinline__ bool pair_init(PairState<Real> &st, unsigned long long p, Real x0, Real v0,
                                          Real q0, const LevelCtx<Real> &L, bool coupled_rt)
{
    const bool coupled = pair_is_coupled<Real, CPL>(coupled_rt);
    st.pair_lo = (uint32_t)p;
    st.word2 = L.word2 ^ (uint32_t)(p >> 32);
    const Real qf = first_flight(L, q0);
    set_start(st, x0);
    st.vf = v0;
    st.i_f = 0;
    st.k = 0;
    st.evc = 0;
    int whole;
    if constexpr (std::is_same<Real, double>::value) {
        const fx::Flight fl = fx::split_flight(fx::pos_of(qf));
        whole = fl.whole;
        st.of = st.oc = q0;
        st.whole_f = st.whole_c = fl.whole;
        st.left_f = st.left_c = fl.left;
    } else {
        st.qf = st.qc = qf;
        whole = st.whole_f = __float2int_rz(qf);
    }
    if (coupled) {
        st.vc = v0;
        st.ic = 0;
        st.num = Real(0);
        st.den = Real(0);
        st.fresh = true;
        if (qf < (Real)L.n) st.Ec = next_coarse_end(L, 0, whole);
    }
    return !(qf < (Real)L.n);
}

// Returns true if the pair has no collision before T (already finished).
template <typename Real, int CPL, int RECIPE = 0>
__device__ __forceinline__ bool pair_start(PairState<Real> &st, unsigned long long p,
                                           const LevelCtx<Real> &L, const PhiloxKeys &keys,
                                           bool coupled_rt)
{
    Real x0, v0, q0;
    pair_start_values<Real, RECIPE>(x0, v0, q0, p, L, keys);
    return pair_init<Real, CPL>(st, p, x0, v0, q0, L, coupled_rt);
}

// One fine event of the FP64 state; returns true when the pair has reached T.
// With every quantity in FP64 the FP64 pipe bounded it (two operations per
// clock and SM), so everything that can be is integer: draws, coefficients, weights and flights are
// positive numbers with 64-bit mantissas (fx::Pos) or fractions, step counts
// and window tests integers.  What is left in FP64 are the sums: 4 operations
// for the position and 6 for the window per fine event and 6 per coarse one,
// against about 45 and 27 before.  At level 8 of the periodic problem (eps = 0.1)
// a fine event with its share of a coarse one takes 92 products of fractions
// and 15 FP64 operations, 11.2 and 8.5 clocks of an SM; 131 071 pairs take
// 1.29 ms, three times that: the pipes share 54 % of the issue slots, and a
// warp waits for its own chain of products (profiles/pair_kernel_fp64_periodic.md).
// FP64 products in place of fx::Pos took 1.86 ms against 1.54 when they went.
template <int CPL, int RECIPE, typename Trace>
__device__ __forceinline__ bool pair_event_fp64(PairState<double> &st, const LevelCtx<double> &L,
                                                const PhiloxKeys &keys, bool coupled_rt, Trace *tr)
{
    typedef Arith<double> A;
    const bool coupled = pair_is_coupled<double, CPL>(coupled_rt);
    const Background<double> &bg = L.bg;
    const DrawFixed d = draw_fixed_r<RECIPE>(st.k + 1u, st.pair_lo, st.word2, L.request, keys);
    const double nu = d.nu_(), chi = d.chi_(), E = fx::to_double(d.E);
    const fx::Pos Rdt = fx::pos_of(bg.Rdt);
    const fx::Pos nu2 = d.nu * d.nu;
    // s = R theta (eq. diffusive-time)
    const Background<double>::Unit f = Background<double>::kd_unit<CPL != 0>(Rdt * fx::steps_left(0, st.left_f), nu2);
    // eq. position-update: nu_k E_k, then nu_{k+1} (1 - e^{-s}) + D chi_k; one
    // rounding at the size of y
    st.xf += fma(st.vf, st.of, fma(f.D, chi, nu * f.om));
    st.i_f += st.whole_f + 1;                                   // eq. time-update
    st.vf = nu;
    st.of = E;
    const fx::Flight fl = fx::split_flight(d.E * fx::pos_of(bg.inv_Rdt));    // eq. intinv (homogeneous)
    st.whole_f = fl.whole;
    st.left_f = fl.left;
    ++st.k;
    if (coupled) {
        if (st.fresh) {
            st.chi_first = chi;
            st.fresh = false;
        }
        st.num = fma(f.beta, chi, st.num);
        st.den = fma(f.beta, f.beta, st.den);
        const int to_end = st.Ec - st.i_f;                      // >= 0
        if (fl.whole < to_end) {
            const double ah = E + f.om;                           // R tau' = R tau + R zeta
            st.num = fma(ah, nu, st.num);
            st.den = fma(ah, ah, st.den);
        } else {
            // coarse KD step
            const fx::Pos sc = Rdt * fx::steps_left(st.Ec - st.ic - st.whole_c - 1, st.left_c);
            const Background<double>::Unit c = Background<double>::kd_unit<false>(sc, nu2);
            const double chit = fx::bits_of(st.den) ? st.num * A::rsqrt_(st.den) : st.chi_first;   // den >= 0
            st.xc += fma(st.vc, st.oc, fma(c.D, chit, nu * c.om));
            // the coarse flight ends at the same collision, to_end steps later.  (The whole
            // steps come from E/(R dt), whose rounding can put to_end R dt above E by an
            // ulp: nothing in a position, but a length that is read out is not negative.)
            st.oc = to_end > 0 ? fma(-fx::from_u32((uint32_t)to_end), bg.Rdt, E) : E;
            st.whole_c = fl.whole - to_end;
            st.left_c = fl.left;
            if constexpr (!std::is_same<Trace, NoTrace>::value)
                tr->coarse(nu, fx::not_negative(st.oc), chit);
            st.ic = st.Ec;
            st.vc = nu;
            ++st.evc;
            if (st.whole_c < L.n - st.ic) st.Ec = next_coarse_end(L, st.ic, st.whole_c);
            st.num = 0.0;
            st.den = 0.0;
            st.fresh = true;
        }
    }
    return !(fl.whole < L.n - st.i_f);
}

// One fine event; returns true when the pair has reached T.
template <typename Real, int CPL, int RECIPE = 0, typename Trace = NoTrace>
__device__ __forceinline__ bool pair_event(PairState<Real> &st, const LevelCtx<Real> &L,
                                           const PhiloxKeys &keys, bool coupled_rt,
                                           Trace *tr = nullptr)
{
    if constexpr (std::is_same<Real, double>::value) {
        return pair_event_fp64<CPL, RECIPE>(st, L, keys, coupled_rt, tr);
    } else {
    typedef Arith<Real> A;
    const bool coupled = pair_is_coupled<Real, CPL>(coupled_rt);
    const Background<Real> &bg = L.bg;
    const Draw<Real> d = draw_r<Real, RECIPE>(st.k + 1u, st.pair_lo, st.word2, L.request, keys);
    const int sq = st.whole_f;                                  // floor: qf >= 0
    const Real theta = bg.dt * ((Real)(sq + 1) - st.qf);        // eq. diffusive-time
    const Real dv = bg.sigma * d.nu;                            // v_{k+1} - mu
    const Real v1 = bg.mu + dv;
    Real a, dd, hs, om;
    bg.kd_coeffs(theta, dv, a, dd, hs, om);
    st.xf = st.xf + st.vf * (st.qf * bg.dt) + (a + dd * d.chi); // eq. position-update
    st.i_f += sq + 1;                                           // eq. time-update
    st.vf = v1;
    st.qf = d.E * bg.inv_Rdt;                                   // eq. intinv (homogeneous)
    // The window and horizon tests compare whole steps: qf < K for an integer
    // K exactly when floor(qf) < K.  (Conversions of step counts run at a
    // quarter of the issue rate; the flight past T saturates.)
    const int whole = __float2int_rz(st.qf);
    st.whole_f = whole;
    ++st.k;

    if (coupled) {
        // Sec. 3.2 aggregation, streamed: this phase's chi with beta, and the
        // new phase's nu with alpha if it collides inside the coarse step.
        Real bh2;
        const Real bh = bg.beta_hat(hs, bh2);
        if (st.fresh) {
            st.chi_first = d.chi;
            st.fresh = false;
        }
        st.num += bh * d.chi;
        st.den += bh2;
        const int to_end = st.Ec - st.i_f;
        if (whole < to_end) {
            const Real ah = st.qf * bg.Rdt + om;                  // R tau' = R tau + R zeta
            st.num += ah * d.nu;
            st.den += ah * ah;
        } else {
            // coarse KD step with nu~ = nu_kappa (eq. nu-update), chi~ (eq.
            // chi-update), then the coarse flight tau~ = fine collision - E_c
            // (homogeneous eq. epsilon-update), carried in fine units.
            const Real thc = bg.dt * ((Real)(st.Ec - st.ic) - st.qc);
            Real ac, dc, hsc, omc;
            bg.kd_coeffs(thc, dv, ac, dc, hsc, omc);
            const Real chit = st.den > Real(0) ? st.num * A::rsqrt_(st.den) : st.chi_first;
            st.xc = st.xc + st.vc * (st.qc * bg.dt) + (ac + dc * chit);
            st.qc = st.qf - (Real)to_end;                         // exact before T
            if constexpr (!std::is_same<Trace, NoTrace>::value)
                tr->coarse(d.nu, st.qc * bg.Rdt, chit);      // nu~, E~ = R tau~, chi~
            st.ic = st.Ec;
            st.vc = v1;
            ++st.evc;
            if (whole - to_end < L.n - st.ic) st.Ec = next_coarse_end(L, st.ic, whole - to_end);
            st.num = Real(0);
            st.den = Real(0);
            st.fresh = true;
        }
    }
    return !(whole < L.n - st.i_f);
    }
}

// Position at T of a path without a collision before T, from the start
// values (heterogeneous backgrounds: v0 is the velocity).
template <typename Real, int PHYS>
__device__ __forceinline__ Real straight_to_T(Real x0, Real v0, const LevelCtx<Real> &L)
{
    if constexpr (PHYS == 0 && std::is_same<Real, double>::value)
        return position_at_T(L, x0, v0 * ((double)L.n * L.bg.Rdt));
    else
        return x0 + v0 * ((Real)L.n * L.bg.dt);          // pair_drift from t = 0
}

// Alg. 1 / Alg. 2 epilogue: move both paths kinetically to T, and leave
// positions x in xf and xc.
template <typename Real, int CPL>
__device__ __forceinline__ void pair_drift(PairState<Real> &st, const LevelCtx<Real> &L, bool coupled_rt)
{
    const bool coupled = pair_is_coupled<Real, CPL>(coupled_rt);
    if constexpr (std::is_same<Real, double>::value) {
        st.xf = position_at_T(L, st.x0, fma(st.vf, (double)max(L.n - st.i_f, 0) * L.bg.Rdt, st.xf));
        if (coupled) st.xc = position_at_T(L, st.x0, fma(st.vc, (double)max(L.n - st.ic, 0) * L.bg.Rdt, st.xc));
        return;
    }
    if (st.i_f < L.n) st.xf = st.xf + st.vf * ((Real)(L.n - st.i_f) * L.bg.dt);
    if (coupled && st.ic < L.n) st.xc = st.xc + st.vc * ((Real)(L.n - st.ic) * L.bg.dt);
}

// ---------------------------------------------------------------------------
// Per-lane sums: Y, Y^2, F(x_f), F(x_f)^2, F(x_c), F(x_c)^2.
//   FP64 mode      : all six in FP64.
//   FP32_DY64 mode : Y and Y^2 formed and summed in FP64 from the FP32 state;
//                    the four F moments as compensated FP32 pairs.
//   FP32_COMP mode : all six as compensated FP32 (sum, error) pairs.
// Compensation is an error-free TwoSum per addition.
// ---------------------------------------------------------------------------
constexpr unsigned kFullMask = 0xffffffffu;

__device__ __forceinline__ void two_sum(float a, float b, float &s, float &e)
{
    s = a + b;
    const float bp = s - a;
    e = (a - (s - bp)) + (b - bp);
}

struct CompF {
    float s, c;
    __device__ void zero() { s = 0.0f; c = 0.0f; }
    __device__ void add(float x) {
        float t, e;
        two_sum(s, x, t, e);
        s = t;
        c += e;
    }
    __device__ void shfl_merge(int off) {
        const float so = __shfl_down_sync(kFullMask, s, off);
        const float co = __shfl_down_sync(kFullMask, c, off);
        float t, e;
        two_sum(s, so, t, e);
        s = t;
        c = c + co + e;
    }
    __device__ double value() const { return (double)s + (double)c; }
};

template <int MODE> struct PairSums;

template <> struct PairSums<kModeFP64> {
    double v[6];
    __device__ void zero() {
#pragma unroll
        for (int j = 0; j < 6; ++j) v[j] = 0.0;
    }
    __device__ void warp_reduce() {
#pragma unroll
        for (int off = 16; off > 0; off >>= 1)
#pragma unroll
            for (int j = 0; j < 6; ++j) v[j] += __shfl_down_sync(kFullMask, v[j], off);
    }
    __device__ double value(int j) const { return v[j]; }
};

template <> struct PairSums<kModeFP32DY64> {
    double sy, sy2;
    CompF q[4];
    __device__ void zero() {
        sy = 0.0;
        sy2 = 0.0;
#pragma unroll
        for (int j = 0; j < 4; ++j) q[j].zero();
    }
    __device__ void warp_reduce() {
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) {
            sy += __shfl_down_sync(kFullMask, sy, off);
            sy2 += __shfl_down_sync(kFullMask, sy2, off);
#pragma unroll
            for (int j = 0; j < 4; ++j) q[j].shfl_merge(off);
        }
    }
    __device__ double value(int j) const { return j == 0 ? sy : j == 1 ? sy2 : q[j - 2].value(); }
};

template <> struct PairSums<kModeFP64U24> : PairSums<kModeFP64> {};

template <> struct PairSums<kModeFP32Comp> {
    CompF q[6];
    __device__ void zero() {
#pragma unroll
        for (int j = 0; j < 6; ++j) q[j].zero();
    }
    __device__ void warp_reduce() {
#pragma unroll
        for (int off = 16; off > 0; off >>= 1)
#pragma unroll
            for (int j = 0; j < 6; ++j) q[j].shfl_merge(off);
    }
    __device__ double value(int j) const { return q[j].value(); }
};

// A lane's running sums.  They change only when a pair finishes, so where the
// event loop needs the registers they live in shared memory; 72 bytes per
// lane keeps bank conflicts at two-way.
template <int MODE> struct LaneSums {
    PairSums<MODE> mom;
    unsigned long long ev_f, ev_c;
    uint32_t pad_[2];
};

// QoI of one finished pair (eq. mlmc-compact): F(x) = x^2 in free space or
// (x mod 1)^2 on the periodic unit interval; Y = F(x_f) - F(x_c), with
// x_f^2 - x_c^2 formed as (x_f - x_c)(x_f + x_c).
__device__ __forceinline__ void add_pair(PairSums<kModeFP64> &ps, double xf, double xc, bool coupled,
                                         bool per)
{
    const double mf = per ? xf - floor(xf) : xf;
    const double mc = per ? xc - floor(xc) : xc;
    const double Ff = mf * mf, Fc = coupled ? mc * mc : 0.0;
    const double y = !coupled ? Ff : per ? Ff - Fc : (xf - xc) * (xf + xc);
    ps.v[0] += y;
    ps.v[1] += y * y;
    ps.v[2] += Ff;
    ps.v[3] += Ff * Ff;
    if (coupled) {
        ps.v[4] += Fc;
        ps.v[5] += Fc * Fc;
    }
}

__device__ __forceinline__ void add_pair(PairSums<kModeFP32DY64> &ps, float xf, float xc, bool coupled,
                                         bool per)
{
    const float mf = per ? xf - floorf(xf) : xf;     // exact in FP32
    const float mc = per ? xc - floorf(xc) : xc;
    const double a = (double)mf, b = (double)mc;
    const double y = !coupled ? a * a : per ? a * a - b * b : (a - b) * (a + b);
    ps.sy += y;
    ps.sy2 += y * y;
    const float Ff = mf * mf, Fc = coupled ? mc * mc : 0.0f;
    ps.q[0].add(Ff);
    ps.q[1].add(Ff * Ff);
    if (coupled) {
        ps.q[2].add(Fc);
        ps.q[3].add(Fc * Fc);
    }
}

__device__ __forceinline__ void add_pair(PairSums<kModeFP32Comp> &ps, float xf, float xc, bool coupled,
                                         bool per)
{
    const float mf = per ? xf - floorf(xf) : xf;
    const float mc = per ? xc - floorf(xc) : xc;
    const float Ff = mf * mf, Fc = coupled ? mc * mc : 0.0f;
    const float y = !coupled ? Ff : per ? Ff - Fc : (xf - xc) * (xf + xc);
    ps.q[0].add(y);
    ps.q[1].add(y * y);
    ps.q[2].add(Ff);
    ps.q[3].add(Ff * Ff);
    if (coupled) {
        ps.q[4].add(Fc);
        ps.q[5].add(Fc * Fc);
    }
}

// Linear QoI F(x) = x (the position at T, the paper's test case): Y = x_f -
// x_c.  fk selects F: 0 x^2, 1 (x mod 1)^2, 2 x.
__device__ __forceinline__ void add_pair_linear(PairSums<kModeFP64> &ps, double xf, double xc, bool coupled)
{
    const double Fc = coupled ? xc : 0.0;
    const double y = xf - Fc;
    ps.v[0] += y;
    ps.v[1] += y * y;
    ps.v[2] += xf;
    ps.v[3] += xf * xf;
    ps.v[4] += Fc;
    ps.v[5] += Fc * Fc;
}

__device__ __forceinline__ void add_pair_linear(PairSums<kModeFP32DY64> &ps, float xf, float xc, bool coupled)
{
    const float Fc = coupled ? xc : 0.0f;
    const double y = (double)xf - (double)Fc;
    ps.sy += y;
    ps.sy2 += y * y;
    ps.q[0].add(xf);
    ps.q[1].add(xf * xf);
    ps.q[2].add(Fc);
    ps.q[3].add(Fc * Fc);
}

__device__ __forceinline__ void add_pair_linear(PairSums<kModeFP32Comp> &ps, float xf, float xc, bool coupled)
{
    const float Fc = coupled ? xc : 0.0f;
    const float y = xf - Fc;
    ps.q[0].add(y);
    ps.q[1].add(y * y);
    ps.q[2].add(xf);
    ps.q[3].add(xf * xf);
    ps.q[4].add(Fc);
    ps.q[5].add(Fc * Fc);
}

template <typename Sums, typename Real>
__device__ __forceinline__ void add_pair_fk(Sums &ps, Real xf, Real xc, bool coupled, int fk)
{
    if (fk == 2)
        add_pair_linear(ps, xf, xc, coupled);
    else
        add_pair(ps, xf, xc, coupled, fk == 1);
}

// Histogram bin: floor((x - lo)/h) inside [lo, hi), else -1; periodic
// positions are first wrapped into [0, 1).  FP64 state divides in FP64; FP32
// state decides its bins in FP32.
struct Bins {
    double lo, hi, h, inv_h;
    float lo_f, hi_f, inv_h_f;
    int nbins;
    bool periodic;
    __device__ int operator()(double x) const {
        if (periodic) x = x - floor(x);
        if (!(x >= lo && x < hi)) return -1;
        // (x - lo)/h decided by the product with 1/h unless that comes within
        // 2^-40 of an integer (an FP64 quotient costs ten products)
        const double q = (x - lo) * inv_h;
        const double t = __dadd_rd(q, 4503599627370496.0);               // 2^52 + floor(q)
        int b = __double2loint(t);
        const double f = q - (t - 4503599627370496.0);
        if (!(f > 0x1p-40 && f < 1.0 - 0x1p-40)) b = (int)floor((x - lo) / h);
        return b < nbins ? b : nbins - 1;
    }
    __device__ int operator()(float x) const {
        if (periodic) x = x - floorf(x);
        if (!(x >= lo_f && x < hi_f)) return -1;
        const int b = (int)floorf((x - lo_f) * inv_h_f);
        return b < nbins ? b : nbins - 1;
    }
};

}  // namespace mlkd
