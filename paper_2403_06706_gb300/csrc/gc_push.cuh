// gc_push.cuh -- the per-particle step of the guiding-centre push (sm_103a): state, evaluation
// phases, events and tally samples, shared by the fused push, the split-step push (gc_push.cu)
// and the push beside the network's evaluation (gc_siren_eval.cu).
#pragma once

#include "gc_device.cuh"
#include "gc_internal.h"

namespace gcp {

// ----------------------------------------------------------------------------------------
// accumulator policy
template <typename T> struct AccOf;
template <> struct AccOf<double> {
    using A = double;
    static __device__ __forceinline__ A from(double d) { return d; }
    static __device__ __forceinline__ double to(A a) { return a; }
    static __device__ __forceinline__ A add(A a, double v) { return a + v; }
    static __device__ __forceinline__ double val(A a) { return a; }
    static __device__ __forceinline__ bool nonpos(A a) { return a <= 0.0; }
};
template <> struct AccOf<float> {
    using A = df;
    static __device__ __forceinline__ A from(double d) { return df_from(d); }
    static __device__ __forceinline__ double to(A a) { return df_to(a); }
    static __device__ __forceinline__ A add(A a, float v) { return df_add(a, v); }
    static __device__ __forceinline__ float val(A a) { return a.hi; }
    static __device__ __forceinline__ bool nonpos(A a) { return a.hi < 0.0f || (a.hi == 0.0f && a.lo <= 0.0f); }
};

// FP32-path uniform from one Philox word: u = (k + 1/2) 2^-31 with k the word's top 31
// bits (the FP64 path's 53-bit draw starts with the same bits, so the two agree to 2^-32),
// together with its complement 1 - u, each with full float relative precision.
struct UPair {
    float u, ub;
};

__device__ __forceinline__ UPair u31(uint32_t w)
{
    const uint32_t k = w >> 1;
    return {fmaf(__uint2float_rn(k), 0x1p-31f, 0x1p-32f),
            fmaf(__uint2float_rn(0x7FFFFFFFu - k), 0x1p-31f, 0x1p-32f)};
}

// -ln(u) without cancellation at either end of (0, 1)
__device__ __forceinline__ float neg_log_u(UPair p) { return p.u < 0.5f ? -logf(p.u) : -log1pf(-p.ub); }

// The same draw as a double pair (a, 1 - a): the member below 1/2 is taken from the float
// that holds it without cancellation and the other is 1 minus it, so the two sum to 1 to
// double rounding (the two floats of a UPair sum to 1 only to float rounding).
struct UPairD {
    double a, b;
};

__device__ __forceinline__ UPairD u31_d(UPair p)
{
    if (p.u < 0.5f) {
        const double a = (double)p.u;
        return {a, 1.0 - a};
    }
    const double b = (double)p.ub;
    return {1.0 - b, b};
}

// FP64 reciprocal and square root by Newton's method from the float estimates, without the
// FP64 division and square-root sequences (GB300's FP64 pipe runs at 1/64 of the FP32 rate,
// and a warp with one colliding lane waits for them). For 0 < x < 3e38: the float estimate
// has a relative error e0 < 2^-21, each Newton step squares it (y <- y + y (1 - x y) for 1/x,
// y <- y + y (1 - x y^2) / 2 for 1/sqrt(x)), so two steps leave e0^4 < 2^-84 and the result
// carries only the FP64 roundings of the steps, a few ulp.
__device__ __forceinline__ double rcp_newton(double x)
{
    double y = (double)__frcp_rn((float)x);
    y = fma(y, fma(-x, y, 1.0), y);
    return fma(y, fma(-x, y, 1.0), y);
}

__device__ __forceinline__ double rsqrt_newton(double x)
{
    double y = (double)rsqrtf((float)x);
    y = fma(0.5 * y, fma(-x * y, y, 1.0), y);
    return fma(0.5 * y, fma(-x * y, y, 1.0), y);
}

__device__ __forceinline__ double sqrt_newton(double x) { return x > 0.0 ? x * rsqrt_newton(x) : 0.0; }

// Time of the end of local step k. Out of line so that the FP64 arithmetic stays in the
// rare branches that need it (rebirth, tally) instead of being hoisted into every step.
static __device__ __noinline__ double step_time(double t0, long long kk, double dt)
{
    return __dadd_rn(t0, __dmul_rn((double)kk, dt));
}

// warp-aggregated increment of base[idx] (idx < 0: no increment for this lane)
__device__ __forceinline__ void agg_inc(uint32_t *base, int idx)
{
    const unsigned mask = __activemask();
    const unsigned grp = __match_any_sync(mask, idx);
    const int leader = __ffs(grp) - 1;
    if (idx >= 0 && (int)(threadIdx.x & 31u) == leader)
        atomicAdd(base + idx, (uint32_t)__popc(grp));
}

__device__ __forceinline__ void agg_inc64(unsigned long long *base, int idx)
{
    const unsigned mask = __activemask();
    const unsigned grp = __match_any_sync(mask, idx);
    const int leader = __ffs(grp) - 1;
    if (idx >= 0 && (int)(threadIdx.x & 31u) == leader)
        atomicAdd(base + idx, (unsigned long long)__popc(grp));
}

// Step of a launch that ends on the next tally sample (the loops run up to the step after it),
// and the one a cadence later: none in this launch where that is beyond an int (a cadence near
// 2^31 stands for "never").
constexpr int kNoTally = INT32_MAX - 1;
__device__ __forceinline__ int after_tally(int next, int cadence)
{
    return cadence < kNoTally - next ? next + cadence : kNoTally;
}

// Snapshot sample of one particle (Sect. 3). FP64: the bins are computed with the same
// operations as the definition (double); FP32: the same formulas in float, with
// gamma - 1 formed without cancellation.
// Out of line: it runs once every cadence steps, and inlined its FP64 bin arithmetic would
// hold registers the step loop needs.
template <typename T>
__device__ __noinline__ void tally_sample(const TallyDev &T_, const PushParams &P, const Phys<T> &ph,
                                             uint32_t e, T x, T y, T z, T u, T mub, T Bm, double age,
                                             uint32_t ncoll, bool take)
{
    int im = -1, iE = -1, ir = -1, ia = -1, ipad = -1;
    unsigned long long s2 = 0;
    if (take) {
        if constexpr (sizeof(T) == 8) {
            const double r = sqrt((double)x * x + (double)y * y + (double)z * z);
            const double gv2 = (double)u * u + 2.0 * (double)mub * (double)Bm / P.m;
            const double gamma = sqrt(1.0 + gv2 / P.c2);
            const double mu = (double)u / sqrt(gv2);
            const double Ek = (gamma - 1.0) * P.m * P.c2;
            const double sin2 = 1.0 - mu * mu;
            im = (int)floor((mu + 1.0) / 2.0 * T_.n_mu);
            if (im >= T_.n_mu) im = T_.n_mu - 1;
            if (im < 0) im = 0;
            const double xe = log(Ek / T_.E_lo) / T_.log_E_ratio * T_.n_E;
            iE = (xe >= 0.0 && xe < T_.n_E) ? (int)floor(xe) : -1;
            const double xr = (r - T_.r_lo) / T_.r_span * T_.n_r;
            ir = (xr >= 0.0 && xr < T_.n_r) ? (int)floor(xr) : -1;
            s2 = (unsigned long long)floor(sin2 * 4294967296.0 + 0.5);
            if (r >= T_.rwin_lo && r < T_.rwin_hi) {
                const double xa = age / T_.age_max * T_.n_age;
                if (xa >= 0.0 && xa < T_.n_age && iE >= 0)
                    ia = (int)(((int64_t)e * T_.n_age + (int)floor(xa)) * T_.n_E + iE);
                if (age < T_.age_young && ncoll >= 1)
                    ipad = (int)e * T_.n_mu + im;
            }
        } else {
            // FP32 path: the same bins from float arithmetic (gamma - 1 without cancellation)
            const float xf = (float)x, yf = (float)y, zf = (float)z, uf = (float)u;
            const float rf = sqrtf(xf * xf + yf * yf + zf * zf);
            const float gv2 = uf * uf + 2.0f * (float)mub * (float)Bm * (float)ph.inv_m;
            const float q = gv2 * (float)ph.inv_c2;
            const float gm1 = q / (sqrtf(1.0f + q) + 1.0f);
            const float muf = uf * rsqrtf(gv2);
            const float Ekf = gm1 * (float)ph.mc2;
            const float s2f = 1.0f - muf * muf;
            im = (int)floorf((muf + 1.0f) * 0.5f * (float)T_.n_mu);
            if (im >= T_.n_mu) im = T_.n_mu - 1;
            if (im < 0) im = 0;
            const float xe = logf(Ekf * T_.inv_E_lo_f) * T_.E_scale_f;
            iE = (xe >= 0.0f && xe < (float)T_.n_E) ? (int)floorf(xe) : -1;
            const float xr = (rf - T_.r_lo_f) * T_.r_scale_f;
            ir = (xr >= 0.0f && xr < (float)T_.n_r) ? (int)floorf(xr) : -1;
            s2 = (unsigned long long)__float2ull_rn(s2f * 4294967296.0f);
            if (rf >= T_.rwin_lo_f && rf < T_.rwin_hi_f) {
                const float agef = (float)age;
                const float xa = agef * T_.age_scale_f;
                if (xa >= 0.0f && xa < (float)T_.n_age && iE >= 0)
                    ia = (int)(((int64_t)e * T_.n_age + (int)floorf(xa)) * T_.n_E + iE);
                if (agef < T_.age_young_f && ncoll >= 1)
                    ipad = (int)e * T_.n_mu + im;
            }
        }
    }
    agg_inc64(T_.n_seen, take ? 0 : -1);
    agg_inc64(T_.n_seen, (take && (iE < 0 || ir < 0)) ? 1 : -1);
    const int ih = (take && iE >= 0 && ir >= 0)
                       ? (int)((((int64_t)e * T_.n_mu + im) * T_.n_E + iE) * T_.n_r + ir)
                       : -1;
    agg_inc(T_.h_mer, ih);
    const int irr = (take && ir >= 0) ? (int)e * T_.n_r + ir : -1;
    agg_inc64(T_.m_cnt, irr);
    if (irr >= 0)
        atomicAdd(T_.m_sin2 + irr, s2);
    agg_inc(T_.h_age, ia);
    agg_inc(T_.h_pad, ipad);
}

// ----------------------------------------------------------------------------------------
// mu_B of the FP32 path is a double-float: the float the right-hand side takes (in the
// particle state) and a low part that only the collision bookkeeping and the launch's load
// and store touch, kept in a per-thread shared-memory slot instead of a register the step
// loop would carry. Blocks of the push kernels have at most kMaxPushBlock threads; the kernel
// that pushes beside the network's evaluation does so in one warp.
constexpr int kMaxPushBlock = 512; // a power of two
__shared__ float s_mub_lo[kMaxPushBlock];

template <typename T>
__device__ __forceinline__ void mub_lo_set(double d, T hi)
{
    if constexpr (sizeof(T) == 4)
        s_mub_lo[threadIdx.x & (kMaxPushBlock - 1)] = (float)(d - (double)hi);
}

template <typename T>
__device__ __forceinline__ double mub_value(T hi)
{
    if constexpr (sizeof(T) == 4)
        return (double)hi + (double)s_mub_lo[threadIdx.x & (kMaxPushBlock - 1)];
    else
        return (double)hi;
}

// ----------------------------------------------------------------------------------------
// Per-particle state and the four evaluation phases of a step, shared by the fused push
// (field evaluated inline) and the split-step push (field samples from a buffer).
//   phase 0  F* at the predictor point (Eq. 5), then the corrector (Eq. 6)
//   phase 1  F^{n+1} at the corrector point, then free path, rebirth and collision tests
//   phase 2  F^n of the new state after a rebirth or collision (start-up, Sect. 2.2)
//   phase 3  F^{n-1} at X^n - dt F^n
// Phases 2-3 run only for the particles that restart.
template <typename T>
struct PState {
    using A = typename AccOf<T>::A;
    A Rx, Ry, Rz, U, S;
    T mub, F0[4], F1[4], vpar0, hprev, Bm0;
    double t_birth;
    uint32_t event, ncoll, flags;
};

// constants of one particle that the step loop reads every step; the rest of its ensemble's
// constants are read from the table where an event needs them
struct PConst {
    float ri2, ro2; // squared shell radii moved 1e-5 inward: beyond them a rebirth is decided in double
    uint32_t e;
};

__device__ __forceinline__ double lambda_of(const PushParams &P, const EnsDev &E)
{
    return P.lambda_override > 0.0 ? P.lambda_override : E.lambda;
}
__device__ __forceinline__ float lambda_f_of(const PushParams &P, const EnsDev &E)
{
    return P.lambda_override > 0.0 ? (float)P.lambda_override : E.lambda_f;
}

// predictor / corrector weights of one step
template <typename T>
struct StepW {
    T a0, a1, c0, cs, c1;
};

template <typename T>
__device__ __forceinline__ void load_particle(const PushParams &P, int64_t i, PConst &c, PState<T> &s)
{
    using Acc = AccOf<T>;
    const int64_t cap = P.st.cap;
    c.e = P.st.ens[i];
    c.ri2 = P.ens[c.e].r_in2 * (1.0f + 1e-5f);
    c.ro2 = P.ens[c.e].r_out2 * (1.0f - 1e-5f);
    s.Rx = Acc::from(P.st.x[i]);
    s.Ry = Acc::from(P.st.y[i]);
    s.Rz = Acc::from(P.st.z[i]);
    s.U = Acc::from(P.st.u[i]);
    s.S = Acc::from(P.st.s_rem[i]);
    s.mub = (T)P.st.mub[i];
    mub_lo_set<T>(P.st.mub[i], s.mub);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        s.F0[k] = (T)P.st.F0[k * cap + i];
        s.F1[k] = (T)P.st.F1[k * cap + i];
    }
    s.vpar0 = (T)P.st.vpar[i];
    s.hprev = (T)P.st.h_prev[i];
    s.t_birth = P.st.t_birth[i];
    s.event = P.st.event[i];
    s.ncoll = P.st.ncoll[i];
    s.flags = P.st.flags[i];
    s.Bm0 = T(0);
}

template <typename T>
__device__ __forceinline__ void store_particle(const PushParams &P, int64_t i, const PState<T> &s)
{
    using Acc = AccOf<T>;
    const int64_t cap = P.st.cap;
    P.st.x[i] = Acc::to(s.Rx);
    P.st.y[i] = Acc::to(s.Ry);
    P.st.z[i] = Acc::to(s.Rz);
    P.st.u[i] = Acc::to(s.U);
    P.st.s_rem[i] = Acc::to(s.S);
    P.st.mub[i] = mub_value<T>(s.mub);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        P.st.F0[k * cap + i] = (double)s.F0[k];
        P.st.F1[k * cap + i] = (double)s.F1[k];
    }
    P.st.vpar[i] = (double)s.vpar0;
    P.st.h_prev[i] = (double)s.hprev;
    P.st.t_birth[i] = s.t_birth;
    P.st.event[i] = s.event;
    P.st.ncoll[i] = s.ncoll;
    if (s.flags != P.st.flags[i]) {
        P.st.flags[i] = s.flags;
        atomicOr(P.gflags, s.flags);
    }
}

// partial stores of the split-step kernels: only what a phase changed, so that the stored
// doubles of untouched fields keep every bit
__device__ __forceinline__ void store_flags(const PushParams &P, int64_t i, uint32_t flags)
{
    if (flags != P.st.flags[i]) {
        P.st.flags[i] = flags;
        atomicOr(P.gflags, flags);
    }
}

template <typename T>
__device__ __forceinline__ void store_RU(const PushParams &P, int64_t i, const PState<T> &s)
{
    using Acc = AccOf<T>;
    P.st.x[i] = Acc::to(s.Rx);
    P.st.y[i] = Acc::to(s.Ry);
    P.st.z[i] = Acc::to(s.Rz);
    P.st.u[i] = Acc::to(s.U);
    store_flags(P, i, s.flags);
}

template <typename T>
__device__ __forceinline__ void store_F(const PushParams &P, int64_t i, const PState<T> &s, int which)
{
    const int64_t cap = P.st.cap;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        if (which == 0)
            P.st.F0[k * cap + i] = (double)s.F0[k];
        else
            P.st.F1[k * cap + i] = (double)s.F1[k];
    }
    if (which == 0) P.st.vpar[i] = (double)s.vpar0;
    store_flags(P, i, s.flags);
}

template <typename T>
__device__ __forceinline__ StepW<T> step_weights(const StepW<T> &w1, T dtT, T hprev)
{
    StepW<T> w = w1;
    if (hprev != dtT) {
        // variable step: tau = dt^n / dt^{n-1}; weights (3+tau)/6,
        // (3+2 tau)/(6(1+tau)), -tau^2/(6(1+tau)) of Eq. 6
        const T tau = dtT / hprev;
        w.a0 = dtT * (T(1) + T(0.5) * tau);
        w.a1 = -dtT * T(0.5) * tau;
        const T q = dtT / (T(6) * (T(1) + tau));
        w.c0 = dtT * (T(3) + tau) / T(6);
        w.cs = q * (T(3) + T(2) * tau);
        w.c1 = -q * tau * tau;
    }
    return w;
}

// the point (R, gamma v_par) at which phase `phase` evaluates the field
template <typename T>
__device__ __forceinline__ void phase_point(int phase, const PState<T> &s, const StepW<T> &w, T dtT, T &px,
                                            T &py, T &pz, T &pu)
{
    using Acc = AccOf<T>;
    px = Acc::val(s.Rx);
    py = Acc::val(s.Ry);
    pz = Acc::val(s.Rz);
    pu = Acc::val(s.U);
    if (phase == 0) {
        px = m_add(px, m_fma(w.a0, s.F0[0], m_mul(w.a1, s.F1[0])));
        py = m_add(py, m_fma(w.a0, s.F0[1], m_mul(w.a1, s.F1[1])));
        pz = m_add(pz, m_fma(w.a0, s.F0[2], m_mul(w.a1, s.F1[2])));
        pu = m_add(pu, m_fma(w.a0, s.F0[3], m_mul(w.a1, s.F1[3])));
    } else if (phase == 3) {
        px = m_fma(-dtT, s.F0[0], px);
        py = m_fma(-dtT, s.F0[1], py);
        pz = m_fma(-dtT, s.F0[2], pz);
        pu = m_fma(-dtT, s.F0[3], pu);
    }
}

// Use the field evaluation Fo (with ax) of phase `phase` for particle slot i; after phase 1
// a rebirth or a collision sets n_phase = 4. kk: index of the step's end time (t_birth on
// rebirth).
// The state a rebirth or a collision changes.
template <typename T>
struct RareState {
    typename AccOf<T>::A Rx, Ry, Rz, U, S;
    T mub;
    double t_birth;
    uint32_t event, ncoll;
};

// A rebirth (Sect. 3) or, if not reborn, a collision (Sect. 2.3) of particle slot i, with B
// magnitude Bm_ and direction (b0, b1, b2) at the new position. Out of line: events are rare,
// and inlined, their FP64 and Philox arithmetic holds registers the step loop needs (the
// ensemble's constants are read from its table here for the same reason).
template <typename T>
__device__ __noinline__ RareState<T> rare_event(const PushParams &P, const Phys<T> &ph, int64_t i, bool reborn,
                                                RareState<T> s, T Bm_, T b0, T b1, T b2, double t0,
                                                long long kk)
{
    using Acc = AccOf<T>;
    const EnsDev &E = P.ens[P.st.ens[i]];
    const uint32_t id = P.st.id[i];
    if (reborn) {
        // Sect. 3: reborn at the injection site with the initial velocity
        const uint4 wd = draw(id, P.seed, s.event++);
        if constexpr (sizeof(T) == 8) {
            s.Rx = E.R0[0];
            s.Ry = E.R0[1];
            s.Rz = E.R0[2];
            s.S = -lambda_of(P, E) * log(u53(wd.z, wd.w));
        } else {
            s.Rx = df{E.R0_hi[0], E.R0_lo[0]};
            s.Ry = df{E.R0_hi[1], E.R0_lo[1]};
            s.Rz = df{E.R0_hi[2], E.R0_lo[2]};
            s.S = df{lambda_f_of(P, E) * neg_log_u(u31(wd.z)), 0.0f};
        }
        s.U = Acc::from(P.st.u_inj[i]);
        s.mub = (T)P.st.mub_inj[i];
        mub_lo_set<T>(P.st.mub_inj[i], s.mub);
        s.ncoll = 0;
        s.t_birth = step_time(t0, kk, P.dt);
    } else {
        // inertial-frame elastic collision: |p| kept, B at R^{n+1}; new pitch
        // cosine from Eq. 10 (mu = 1 - 2a) or Eq. 12 (mu = +-sqrt(a))
        const uint4 wd = draw(id, P.seed, s.event++);
        if constexpr (sizeof(T) == 8) {
            const double a = u53(wd.x, wd.y);
            const double mu_new = (E.scatter_law == 0) ? 1.0 - 2.0 * a : ((wd.x & 1u) ? -sqrt(a) : sqrt(a));
            const double Bm = (double)Bm_;
            const double uu = Acc::to(s.U);
            if (P.wind_u > 0.0) {
                // Sect. 3.2: elastic in the frame of the wind u = wind_u R/r; the guiding
                // centre drifts with u_perp already, so the frame change is a boost along
                // b by V = u.b (p_perp unchanged): u~ = gV (u - V gamma), back with -V
                const double X = Acc::to(s.Rx), Y = Acc::to(s.Ry), Z = Acc::to(s.Rz);
                const double V = P.wind_u * (X * b0 + Y * b1 + Z * b2) /
                                 sqrt(X * X + Y * Y + Z * Z);
                const double gV = 1.0 / sqrt(1.0 - V * V / P.c2);
                const double pp2 = 2.0 * (double)s.mub * Bm / P.m;
                const double gam = sqrt(1.0 + (uu * uu + pp2) / P.c2);
                const double ut = gV * (uu - V * gam);
                const double pt2 = ut * ut + pp2;
                const double gt = sqrt(1.0 + pt2 / P.c2);
                s.U = gV * (mu_new * sqrt(pt2) + V * gt);
                s.mub = (1.0 - mu_new * mu_new) * pt2 * P.m / (2.0 * Bm);
            } else {
                const double pm2 = uu * uu + 2.0 * (double)s.mub * Bm / P.m;
                const double pm = sqrt(pm2);
                s.U = mu_new * pm;
                s.mub = (1.0 - mu_new * mu_new) * pm2 * P.m / (2.0 * Bm);
            }
            if (P.collision_form == 0)
                s.S = -lambda_of(P, E) * log(u53(wd.z, wd.w));
        } else {
            // FP32 path: the pitch is drawn from float uniforms, the momentum bookkeeping
            // runs in FP64 on the double-float gamma v_par and mu_B, so |p| (|p~| in the wind
            // frame) is kept to double-float rounding (~1e-14), not FP32's; mu^2 + sin^2 = 1
            // to FP64 rounding (u31_d), and 1/x, sqrt(x) come from Newton steps.
            const UPairD ua = u31_d(u31(wd.x));
            double mu_new, sin2;
            if (E.scatter_law == 0) {
                mu_new = ua.b - ua.a; // Eq. 10: mu = (1 - a) - a
                sin2 = 4.0 * ua.a * ua.b;
            } else {
                const double su = sqrt_newton(ua.a); // Eq. 12: mu^2 = a
                mu_new = (wd.x & 1u) ? -su : su;
                sin2 = ua.b;
            }
            const double K = (double)Bm_ * P.two_over_m; // (p_perp / m)^2 = mu_B K
            const double uu = Acc::to(s.U);
            const double pp2 = mub_value<T>(s.mub) * K;
            double pm2 = uu * uu + pp2, un;
            if (P.wind_u > 0.0) {
                // the wind-frame collision of the FP64 branch above
                const double X = Acc::to(s.Rx), Y = Acc::to(s.Ry), Z = Acc::to(s.Rz);
                const double V = P.wind_u * (X * (double)b0 + Y * (double)b1 + Z * (double)b2) *
                                 rsqrt_newton(X * X + Y * Y + Z * Z);
                const double gV = rsqrt_newton(1.0 - V * V * P.inv_c2);
                const double gam = sqrt_newton(1.0 + pm2 * P.inv_c2);
                const double ut = gV * (uu - V * gam);
                pm2 = ut * ut + pp2;
                const double gt = sqrt_newton(1.0 + pm2 * P.inv_c2);
                un = gV * (mu_new * sqrt_newton(pm2) + V * gt);
            } else {
                un = mu_new * sqrt_newton(pm2);
            }
            const double mub_new = sin2 * pm2 * rcp_newton(K);
            s.U = Acc::from(un);
            s.mub = (T)mub_new;
            mub_lo_set<T>(mub_new, s.mub);
            if (P.collision_form == 0)
                s.S = df{lambda_f_of(P, E) * neg_log_u(u31(wd.z)), 0.0f};
        }
        ++s.ncoll;
    }
    return s;
}

template <typename T>
__device__ __forceinline__ void phase_consume(int phase, int &n_phase, int64_t i, PState<T> &s, const PConst &c,
                                              const T Fo[4],
                                              const Aux<T> &ax, const StepW<T> &w, const PushParams &P,
                                              const Phys<T> &ph, T dtT, double t0, long long kk,
                                              unsigned &n_coll, unsigned &n_reb)
{
    using Acc = AccOf<T>;
    if (phase == 0) {
        s.Rx = Acc::add(s.Rx, m_fma(w.c1, s.F1[0], m_fma(w.c0, s.F0[0], m_mul(w.cs, Fo[0]))));
        s.Ry = Acc::add(s.Ry, m_fma(w.c1, s.F1[1], m_fma(w.c0, s.F0[1], m_mul(w.cs, Fo[1]))));
        s.Rz = Acc::add(s.Rz, m_fma(w.c1, s.F1[2], m_fma(w.c0, s.F0[2], m_mul(w.cs, Fo[2]))));
        s.U = Acc::add(s.U, m_fma(w.c1, s.F1[3], m_fma(w.c0, s.F0[3], m_mul(w.cs, Fo[3]))));
    } else if (phase == 1) {
        const T px = Acc::val(s.Rx), py = Acc::val(s.Ry), pz = Acc::val(s.Rz);
        // Sect. 2.3: path length along B in this step
        const T ds = dtT * (fabs(s.vpar0) + fabs(ax.vpar)) * T(0.5);
        bool collide = false;
        if (!P.no_scatter) {
            if (P.collision_form == 0) {
                s.S = Acc::add(s.S, -ds);
                collide = Acc::nonpos(s.S);
            } else {
                // the per-step draw of Eq. 9: collide if a < 1 - exp(-ds / lambda)
                const uint4 wd = draw(P.st.id[i], P.seed, s.event++);
                if constexpr (sizeof(T) == 8)
                    collide = u53(wd.x, wd.y) < 1.0 - exp(-(double)ds / lambda_of(P, P.ens[c.e]));
                else
                    collide = u31(wd.x).u < -expm1f(-(float)ds / lambda_f_of(P, P.ens[c.e]));
            }
        }
        bool reborn = false;
        if (!P.no_rebirth) {
            if (sizeof(T) == 8) {
                const double xx = Acc::to(s.Rx), yy = Acc::to(s.Ry), zz = Acc::to(s.Rz);
                const double r1 = sqrt(xx * xx + yy * yy + zz * zz);
                reborn = (r1 < P.ens[c.e].r_in || r1 > P.ens[c.e].r_out);
            } else {
                const float xx = (float)px, yy = (float)py, zz = (float)pz;
                const float r2 = xx * xx + yy * yy + zz * zz;
                if (r2 < c.ri2 || r2 > c.ro2) {
                    // near or beyond the shell: decide in double from the accumulated position
                    const double X = Acc::to(s.Rx), Y = Acc::to(s.Ry), Z = Acc::to(s.Rz);
                    const double r1 = sqrt(X * X + Y * Y + Z * Z);
                    reborn = (r1 < P.ens[c.e].r_in || r1 > P.ens[c.e].r_out);
                }
            }
        }
        if (reborn || collide) {
            RareState<T> o{s.Rx, s.Ry, s.Rz, s.U, s.S, s.mub, s.t_birth, s.event, s.ncoll};
            o = rare_event<T>(P, ph, i, reborn, o, ax.Bm, ax.b[0], ax.b[1], ax.b[2], t0, kk);
            s.Rx = o.Rx; s.Ry = o.Ry; s.Rz = o.Rz; s.U = o.U; s.S = o.S;
            s.mub = o.mub; s.t_birth = o.t_birth; s.event = o.event; s.ncoll = o.ncoll;
            if (reborn)
                ++n_reb;
            else
                ++n_coll;
            n_phase = 4;
        } else {
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                s.F1[k] = s.F0[k];
                s.F0[k] = Fo[k];
            }
            s.vpar0 = ax.vpar;
            s.Bm0 = ax.Bm;
        }
    } else if (phase == 2) {
#pragma unroll
        for (int k = 0; k < 4; ++k)
            s.F0[k] = Fo[k];
        s.vpar0 = ax.vpar;
        s.Bm0 = ax.Bm;
    } else {
#pragma unroll
        for (int k = 0; k < 4; ++k)
            s.F1[k] = Fo[k];
    }
}
// ----------------------------------------------------------------------------------------
// Field evaluations outside the step: samples of the requested points.
// sample k of S, in global (read-only) or shared memory
template <bool SHARED = false>
__device__ __forceinline__ void load_sample(const float *S, int64_t k, int g_in, Sample<float> &s)
{
    const float4 *q = reinterpret_cast<const float4 *>(S + k * kSampleStride);
    float v[40];
#pragma unroll
    for (int j = 0; j < 10; ++j) {
        const float4 t = SHARED ? q[j] : __ldg(q + j);
        v[4 * j] = t.x;
        v[4 * j + 1] = t.y;
        v[4 * j + 2] = t.z;
        v[4 * j + 3] = t.w;
    }
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        s.B[c] = v[c];
        s.E[c] = v[3 + c];
        s.dPhi[c] = v[34 + c];
    }
#pragma unroll
    for (int d = 0; d < 3; ++d)
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            s.dB[d][c] = v[6 + 3 * d + c];
            s.dE[d][c] = v[15 + 3 * d + c];
            s.g[d][c] = g_in ? v[24 + 3 * d + c] : (d == c ? 1.0f : 0.0f);
        }
    s.flags = g_in ? __float_as_uint(v[33]) : 0u;
}

__device__ __forceinline__ void flush_counters(const PushParams &P, unsigned n_coll, unsigned n_reb)
{
    const unsigned mask = __activemask();
    const unsigned c_sum = __reduce_add_sync(mask, n_coll);
    const unsigned r_sum = __reduce_add_sync(mask, n_reb);
    if ((threadIdx.x & 31u) == (unsigned)(__ffs(mask) - 1)) {
        if (c_sum) atomicAdd(P.counters + 0, (unsigned long long)c_sum);
        if (r_sum) atomicAdd(P.counters + 1, (unsigned long long)r_sum);
    }
}

// One evaluation phase of a particle whose field is sampled elsewhere: sample smp of its
// request, taken in phase `phase` of step `step` (of n_steps; kk: index of that step's end
// time, step0: the call's first step). Leaves phase and step at the next request and that
// request in px, py, pz; returns what has changed: 0 R and u; 1 the step's bookkeeping; 2 all
// (an event); 3 F^n; 4 F^{n-1}.
enum : int { CHANGED_RU = 0, CHANGED_STEP, CHANGED_ALL, CHANGED_F0, CHANGED_F1 };

__device__ __forceinline__ int sampled_phase(const PushParams &P, const Phys<float> &ph, int ideal, int64_t i,
                                             PState<float> &s, const PConst &c, const Sample<float> &smp,
                                             const StepW<float> &w1, float dtT, long long kbase, int &step, int &phase,
                                             float &px, float &py, float &pz, unsigned &n_coll, unsigned &n_reb)
{
    using Acc = AccOf<float>;
    const long long kk = kbase + step + 1;
    const StepW<float> w = step_weights(w1, dtT, s.hprev);
    float Fo[4], pu;
    Aux<float> ax;
    int n_phase = 2, changed;
    auto tally = [&]() {
        if (P.tally_on && (P.step0 + kk) % P.tally.cadence == 0) {
            const double t_new = step_time(P.t0, kk, P.dt);
            tally_sample<float>(P.tally, P, ph, c.e, Acc::val(s.Rx), Acc::val(s.Ry), Acc::val(s.Rz), Acc::val(s.U),
                                s.mub, s.Bm0, t_new - s.t_birth, s.ncoll,
                                s.t_birth >= P.tally.t_start && (int)c.e < P.tally.n_ens);
        }
    };
    s.flags |= smp.flags;
    bool ends = false; // the step is complete
    if (phase == 0) {
        phase_point(0, s, w, dtT, px, py, pz, pu);
        rhs(smp, ph, ideal, pu, s.mub, Fo, ax);
        phase_consume(0, n_phase, i, s, c, Fo, ax, w, P, ph, dtT, P.t0, kk, n_coll, n_reb);
        px = Acc::val(s.Rx);
        py = Acc::val(s.Ry);
        pz = Acc::val(s.Rz);
        changed = CHANGED_RU;
        phase = 1;
    } else if (phase == 1) {
        phase_point(1, s, w, dtT, px, py, pz, pu);
        rhs(smp, ph, ideal, pu, s.mub, Fo, ax);
        phase_consume(1, n_phase, i, s, c, Fo, ax, w, P, ph, dtT, P.t0, kk, n_coll, n_reb);
        s.hprev = dtT;
        if (n_phase == 4) {
            px = Acc::val(s.Rx);
            py = Acc::val(s.Ry);
            pz = Acc::val(s.Rz);
            changed = CHANGED_ALL;
            phase = 2;
        } else {
            if (!(m_finite(Acc::val(s.Rx)) && m_finite(Acc::val(s.U)) && m_finite(s.F0[0])))
                s.flags |= FLAG_NONFINITE;
            tally();
            changed = CHANGED_STEP;
            ends = true;
        }
    } else if (phase == 2) {
        phase_point(2, s, w, dtT, px, py, pz, pu);
        rhs(smp, ph, ideal, pu, s.mub, Fo, ax);
        phase_consume(2, n_phase, i, s, c, Fo, ax, w, P, ph, dtT, P.t0, kk, n_coll, n_reb);
        tally();
        phase_point(3, s, w, dtT, px, py, pz, pu);
        changed = CHANGED_F0;
        phase = 3;
    } else {
        phase_point(3, s, w, dtT, px, py, pz, pu);
        rhs(smp, ph, ideal, pu, s.mub, Fo, ax);
        phase_consume(3, n_phase, i, s, c, Fo, ax, w, P, ph, dtT, P.t0, kk, n_coll, n_reb);
        if (!(m_finite(Acc::val(s.Rx)) && m_finite(Acc::val(s.U)) && m_finite(s.F0[0])))
            s.flags |= FLAG_NONFINITE;
        changed = CHANGED_F1;
        ends = true;
    }
    if (ends) {
        // the next step's predictor point
        ++step;
        phase = 0;
        phase_point(0, s, step_weights(w1, dtT, s.hprev), dtT, px, py, pz, pu);
    }
    return changed;
}

template <typename T>
static Phys<T> make_phys(const PhysHost &p)
{
    Phys<T> q;
    q.qm = (T)p.qm;
    q.inv_qm = (T)(1.0 / p.qm);
    q.inv_m = (T)p.inv_m;
    q.inv_c2 = (T)p.inv_c2;
    q.mc2 = (T)(1.0 / (p.inv_m * p.inv_c2));
    q.drift_mask = p.drift_mask;
    return q;
}

} // namespace gcp
