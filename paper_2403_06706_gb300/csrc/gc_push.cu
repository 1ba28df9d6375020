// gc_push.cu -- persistent guiding-centre push and injection kernels (sm_103a).
//
// One thread (in FP64, for few particles, four lanes) owns one particle at a time and keeps its
// whole state in registers for all the steps of a launch. Per step (Sect. 2.2):
//   predictor X* (Eq. 5) -> F* = F(X*) -> corrector X^{n+1} (Eq. 6) -> F^{n+1}
//   -> free path decrement by dt (|v_par^n| + |v_par^{n+1}|)/2 (Sect. 2.3, Eq. 9)
//   -> rebirth if the particle left [r_in, r_out], else a collision if the free path is
//      used up (new pitch cosine from Eq. 10 or Eq. 12, |p| kept; inertial frame, Sect. 3)
//   -> backward-Euler start-up of the history after either (Sect. 2.2)
//   -> every `cadence` steps a snapshot sample into the tallies (Sect. 3).
//
// Precision: GC_PREC_FP64 runs everything in double. GC_PREC_FP32_MIXED evaluates the
// field and Eqs. 1-2 in float and accumulates R, gamma v_par and the free path in
// double-float pairs; mu_B is a double-float too (the right-hand side takes its float
// part), and the rare collision and rebirth updates of gamma v_par and mu_B run in double.
#include <algorithm>
#include <type_traits>

#include "gc_push.cuh"

namespace gcp {

// ----------------------------------------------------------------------------------------
// Threads of the push resident per SM, which its register budget (65536 / threads) allows and
// one block may hold. FP32: 512 (640 at 96 registers spill 48 bytes and measured 1.5 % slower,
// also with the rarely used state in shared memory; 384 for the potential channel 5 % slower);
// time-dependent fields 384 (512 spilled 172 bytes and measured 6 % slower). FP64: 256 (384
// and 512 spill and measured 0.4 % and 1.7 % slower: the FP64 pipe, not latency, bounds it).
template <typename T, bool TD>
constexpr int kPushThreads = sizeof(T) == 4 ? (TD ? 384 : 512) : 256;

// Particles of a partial round that a block takes at a time (see push_kernel).
template <typename T>
constexpr unsigned kSpread = sizeof(T) == 8 ? 32 : 128;

// Fused push: one thread owns a particle for all the steps of a launch and evaluates the
// grid field inline.
template <typename T, bool TD, int POT>
__global__ void __launch_bounds__((kPushThreads<T, TD>), 1) push_kernel(const __grid_constant__ GridMeta<T> gm, const __grid_constant__ Phys<T> ph,
                                                   const __grid_constant__ PushParams P)
{
    unsigned n_coll = 0, n_reb = 0;
    const T dtT = (T)P.dt;
    double t0 = P.t0;
    int64_t step0 = P.step0;
    if (P.clock) {
        t0 = P.clock[0];
        step0 = (int64_t)P.clock[1] + P.kbase;
    }
    // Eq. 5-6 weights at tau = 1: 3/2, -1/2 (AB2) and 2/3, 5/12, -1/12 (AM3)
    const StepW<T> w1 = {dtT * T(1.5), dtT * T(-0.5), dtT * T(2.0 / 3.0), dtT * T(5.0 / 12.0),
                         dtT * T(-1.0 / 12.0)};
    // time-dependent fields: time of the call's start after the first snapshot
    const T tr0 = TD ? (T)(t0 - gm.t_snap0) : T(0);
    // the two phases of a step as straight-line code (each with its own copy of the field
    // evaluation) in the steady-field kernels; the time-dependent ones keep one copy in a
    // loop over the phases (unrolled, they spill)
    constexpr bool kUnrollPhases = !TD;

    // Particles of the full rounds in blocks of neighbours (which share cells); those left from
    // P.spread_from on, all of a small population, in groups of kSpread<T>, one per block in turn:
    // a partial round then has its warps on all SMs. (With whole blocks 200 000 particles, 2.57
    // rounds of one block of 512 per SM, ran 11 % slower than with blocks of 128; groups of 32
    // instead of 128 3 % slower, but 8 % faster in FP64 where an SM gets fewer than four warps.)
    constexpr unsigned group = kSpread<T>;
    int64_t next = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    for (;;) {
        if (next >= P.spread_from)
            next = P.spread_from + ((int64_t)(threadIdx.x / group) * gridDim.x + blockIdx.x) * group + threadIdx.x % group;
        if (next >= P.st.n)
            break;
        const uint32_t i = (uint32_t)next; // ids, and so slots, have 32 bits
        PConst c;
        PState<T> s;
        load_particle(P, i, c, s);
        int next_tally = kNoTally; // the step that ends on the next tally sample
        if (P.tally_on) {
            const int64_t K = P.tally.cadence;
            next_tally = (int)((K - 1 - (step0 % K)) % K);
        }

        // One iteration evaluates the field at two points: a step's predictor and corrector
        // points or, for a particle whose step ended in a rebirth or a collision, the two points
        // of its start-up history (Sect. 2.2). Such a particle takes an iteration more than its
        // neighbours in the warp and keeps its own step count, up to the next tally sample,
        // which the warp takes together. Restarting out of line instead, the warp made two more
        // evaluations for one lane in every step in which any of the 32 had an event (3.5 % of
        // the steps at lambda = 0.1 to 1 AU, 8 % at 0.1 AU).
        int k = 0;
        do {
            const int k_end = min(P.n_steps, next_tally + 1);
            bool restart = false;
            while (k < k_end) {
                const StepW<T> w = step_weights(w1, dtT, s.hprev);
                // the predictor, corrector and restart evaluations are at the step's end time,
                // the start-up's F^{n-1} one step earlier
                const T t_end = TD ? tr0 + (T)(P.kbase + k + 1) * dtT : T(0);
                int n_phase = 2;
                // phase 0: predictor point and corrector; phase 1: F^{n+1}, free path, events. A
                // restarting particle has F^n = F^{n-1} = 0, so that its predictor point is the
                // state itself
                auto run_phase = [&](auto kind, int phase) {
                    constexpr int EV = decltype(kind)::value;
                    T px, py, pz, pu;
                    phase_point(phase, s, w, dtT, px, py, pz, pu);
                    if (phase == 1 && restart) phase_point(3, s, w, dtT, px, py, pz, pu);
                    T Fo[4];
                    Aux<T> ax;
                    s.flags |= eval_F<T, TD, POT, EV>(gm, ph, px, py, pz, pu, s.mub, Fo, ax,
                                                      TD && phase == 1 && restart ? t_end - dtT : t_end, restart);
                    if (restart)
                        phase_consume(phase + 2, n_phase, i, s, c, Fo, ax, w, P, ph, dtT, t0, 0, n_coll, n_reb);
                    else
                        phase_consume(phase, n_phase, i, s, c, Fo, ax, w, P, ph, dtT, t0,
                                      (long long)(P.kbase + k + 1), n_coll, n_reb);
                };
                using std::integral_constant;
                if constexpr (kUnrollPhases) {
                    run_phase(integral_constant<int, EV_PREDICTOR>{}, 0);
                    run_phase(integral_constant<int, EV_CORRECTOR>{}, 1);
                } else {
#pragma unroll 1
                    for (int phase = 0; phase < 2; ++phase)
                        run_phase(integral_constant<int, EV_PREDICTOR>{}, phase);
                }
                if (n_phase == 4) {
#pragma unroll
                    for (int q = 0; q < 4; ++q)
                        s.F0[q] = s.F1[q] = T(0);
                    restart = true;
                    continue;
                }
                restart = false;
                s.hprev = dtT;
                ++k;
            }
            if (k == next_tally + 1) {
                next_tally = after_tally(next_tally, P.tally.cadence);
                const double t_new = step_time(t0, (long long)(P.kbase + k), P.dt);
                tally_sample<T>(P.tally, P, ph, c.e, AccOf<T>::val(s.Rx), AccOf<T>::val(s.Ry), AccOf<T>::val(s.Rz),
                                AccOf<T>::val(s.U), s.mub, s.Bm0, t_new - s.t_birth, s.ncoll,
                                s.t_birth >= P.tally.t_start && (int)c.e < P.tally.n_ens);
            }
        } while (k < P.n_steps);
        // a non-finite position is flagged by the gather at the next evaluation; what the last
        // step leaves is checked here
        if (!(m_finite(AccOf<T>::val(s.Rx)) && m_finite(AccOf<T>::val(s.U)) && m_finite(s.F0[0])))
            s.flags |= FLAG_NONFINITE;
        store_particle(P, i, s);
        if (i >= P.spread_from)
            break;
        next = (int64_t)i + (int64_t)gridDim.x * blockDim.x;
    }
    // counters: one atomic per warp
    const unsigned mask = __activemask();
    const unsigned c_sum = __reduce_add_sync(mask, n_coll);
    const unsigned r_sum = __reduce_add_sync(mask, n_reb);
    if ((threadIdx.x & 31u) == (unsigned)(__ffs(mask) - 1)) {
        if (c_sum) atomicAdd(P.counters + 0, (unsigned long long)c_sum);
        if (r_sum) atomicAdd(P.counters + 1, (unsigned long long)r_sum);
    }
}

// ----------------------------------------------------------------------------------------
// FP64 push of a small population: four lanes per particle. An FP64 instruction holds its
// scheduler's pipe for 64 cycles whatever the number of active lanes, so with fewer particles
// than lanes the time is the number of instructions in a particle's chain, which spreading the
// particles thinner does not shorten. Lane c = 0, 1, 2 of a quad holds component c of every
// vector (and the channels B_c, E_c of the gather), lane 3 gamma v_par and the potential;
// products over components and cross products go through shuffles, the polar angles and the
// roots of the two radii are taken in different lanes at once, scalars are carried by all four.
// Rounding for rounding what push_kernel does, so that the launch's shape and the size of the
// population don't show in the results. 400 steps, E_par = 0, one particle per lane -> this:
// 608 to 2432 particles 10.15 -> 5.9 ms, 4864 6.3 ms, 7296 8.4, 9728 10.9 (from four warps
// per SM on the pipe is shared, and the work common to the lanes counts): push_quad_fits.
__device__ __forceinline__ double q_get(double v, int src) { return __shfl_sync(0xffffffffu, v, src, 4); }

// dot3 of two vectors held by lanes 0-2: the chain of its three roundings goes round the lanes
__device__ __forceinline__ double q_dot(double a, double b)
{
    double t = a * b;
    t = m_fma(a, b, q_get(t, 1));
    t = m_fma(a, b, q_get(t, 0));
    return q_get(t, 2);
}

// component c of cross3: a1, a2 and b1, b2 are the next two components
__device__ __forceinline__ double q_cross(double a1, double a2, double b1, double b2) { return m_fma(a1, b2, -m_mul(a2, b1)); }

struct QuadEval {
    double F;           // this lane's component of (F_x, F_y, F_z, F_u)
    double vpar, Bm, b; // b: this lane's component
    double r2;          // squared radius of the point
    uint32_t flags;
};

// Eqs. 1-3 at the point whose component (x, y, z, gamma v_par) this lane holds in p: gather and
// rhs, rounding for rounding
template <int POT, int EV>
__device__ __forceinline__ QuadEval quad_eval(const GridMeta<double> &gm, const Phys<double> &ph, int c, double p, double mub,
                                              bool other)
{
    QuadEval o;
    const int c1 = (c + 1) % 3, c2 = (c + 2) % 3; // the next components, cyclically (lane 3: any)
    const double x = q_get(p, 0), y = q_get(p, 1), z = q_get(p, 2), u = q_get(p, 3);
    uint32_t flags = 0;
    double rho2 = other ? m_fma(x, x, m_mul(y, y)) : m_fma(y, y, m_mul(x, x));
    if (!(rho2 > 1e-30)) {
        flags |= FLAG_AXIS;
        rho2 = 1e-30;
    }
    const double r2 = EV == EV_CORRECTOR && POT != POT_ON && !other ? m_add(rho2, m_mul(z, z)) : m_fma(z, z, rho2);
    const double inv = m_rsqrt(c == 0 ? rho2 : r2);
    const double inv_rho = q_get(inv, 0), inv_r = q_get(inv, 1);
    const double rho = rho2 * inv_rho;
    // index coordinates: lane 0 theta, lane 1 phi, lane 2 r
    const double X = c == 0 ? z : x, Y = c == 0 ? rho : y;
    double ang = refine_angle(X, Y, c == 0 ? inv_r : inv_rho, m_atan2((float)Y, (float)X));
    if (c == 1 && ang < 0.0) ang += two_pi<double>();
    double q = c == 2 ? m_mul(m_fma(r2, inv_r, -gm.r_min), gm.inv_dr) : ang * (c == 0 ? gm.inv_dth : gm.inv_dph);
    const unsigned lane0 = threadIdx.x & 28u;
    if ((__ballot_sync(0xffffffffu, !m_finite(q)) >> lane0) & 7u) {
        flags |= FLAG_NONFINITE;
        q = 0.0;
    }
    const double fl = floor(q);
    int idx = (int)fl;
    double f = q - fl;
    const int last = c == 2 ? gm.n_r - 2 : gm.n_th - 2;
    const bool out = c == 2 && (q < -1.0 || q > gm.n_r);
    if ((__ballot_sync(0xffffffffu, out) >> lane0) & 4u) flags |= FLAG_OUT_OF_GRID;
    if (c == 1) {
        if (idx >= gm.n_ph) idx -= gm.n_ph;
    } else if (idx < 0 || idx > last) {
        f = idx < 0 ? 0.0 : 1.0;
        idx = idx < 0 ? 0 : last;
    }
    const int i = __shfl_sync(0xffffffffu, idx, 2, 4), j = __shfl_sync(0xffffffffu, idx, 0, 4),
              k = __shfl_sync(0xffffffffu, idx, 1, 4);
    const double fr = q_get(f, 2), ft = q_get(f, 0), fp = q_get(f, 1);
    const int kn = k + 1 == gm.n_ph ? 0 : k + 1;

    // channels B_c and E_c (lane 3: the potential, and E_x unused)
    const uint32_t nr8 = (uint32_t)gm.n_r * 8u;
    const uint32_t o0 = (((uint32_t)k * (uint32_t)gm.n_th + (uint32_t)j) * (uint32_t)gm.n_r + (uint32_t)i) * 8u;
    const uint32_t o1 = (((uint32_t)kn * (uint32_t)gm.n_th + (uint32_t)j) * (uint32_t)gm.n_r + (uint32_t)i) * 8u;
    double val[2], d[2][3];
#pragma unroll
    for (int ch = 0; ch < 2; ++ch) {
        const double *nodes = gm.nodes + (ch == 0 ? (c < 3 ? c : 7) : 3 + (c < 3 ? c : 0));
        double L[2][2], D[2][2];
#pragma unroll
        for (int cc = 0; cc < 2; ++cc)
#pragma unroll
            for (int b = 0; b < 2; ++b) {
                const double *n0 = nodes + (cc ? o1 : o0) + (b ? nr8 : 0u);
                const double v0 = __ldg(n0), v1 = __ldg(n0 + 8);
                D[b][cc] = v1 - v0;
                L[b][cc] = v0 + fr * D[b][cc];
            }
        double V[2], Dr[2], Dt[2];
#pragma unroll
        for (int cc = 0; cc < 2; ++cc) {
            Dt[cc] = L[1][cc] - L[0][cc];
            V[cc] = L[0][cc] + ft * Dt[cc];
            Dr[cc] = D[0][cc] + ft * (D[1][cc] - D[0][cc]);
        }
        d[ch][2] = V[1] - V[0];
        val[ch] = V[0] + fp * d[ch][2];
        d[ch][0] = Dr[0] + fp * (Dr[1] - Dr[0]);
        d[ch][1] = Dt[0] + fp * (Dt[1] - Dt[0]);
    }
    const double B = val[0], E = val[1];
    // this lane's component of the index coordinates' gradients (see gather)
    const double st = inv_r * inv_r * gm.inv_dth, sp = inv_rho * inv_rho * gm.inv_dph;
    double g[3];
    g[0] = p * (inv_r * gm.inv_dr);
    g[1] = (c < 2 ? z * inv_rho * p : -rho) * st;
    g[2] = c == 0 ? -y * sp : (c == 1 ? x * sp : 0.0);

    // the right-hand side
    const double B2 = q_dot(B, B);
    const double inv_B = m_rsqrt(B2), Bm = B2 * inv_B, inv_B2 = inv_B * inv_B, b = B * inv_B;
    double sb[3];
#pragma unroll
    for (int a = 0; a < 3; ++a)
        sb[a] = q_dot(d[0][a], b);
    const double gB01 = m_fma(sb[0], g[0], m_mul(sb[1], g[1]));
    const double gB = c == 2 ? gB01 : m_fma(sb[2], g[2], gB01);
    const double b_gB = q_dot(b, gB);
    const double B1 = q_get(B, c1), Bq = q_get(B, c2), E1 = q_get(E, c1), Eq = q_get(E, c2);
    const double vE = q_cross(E1, Eq, B1, Bq) * inv_B2;
    double Epar = 0.0;
    if constexpr (POT == POT_ON) {
        double pb[3], dPhi[3];
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            pb[a] = q_dot(g[a], b);
            dPhi[a] = q_get(d[0][a], 3);
        }
        Epar = -dot3(dPhi, pb);
    } else if constexpr (POT == POT_NONE) {
        Epar = q_dot(E, b);
    }
    const double g2 = m_fma(m_fma(u, u, m_mul(2.0 * mub * Bm, ph.inv_m)), ph.inv_c2, 1.0);
    const double inv_g = m_rsqrt(g2), gamma = g2 * inv_g, vpar = u * inv_g;
    const double mirror = m_mul(mub * ph.inv_m * inv_g, b_gB);
    double F, Fu;
    if (ph.drift_mask == 1) {
        F = vpar * b;
        Fu = POT == POT_IDEAL ? -mirror : m_fma(ph.qm, Epar, -mirror);
    } else {
        const double wv = m_fma(vpar, b, vE);
        double pw[3];
        pw[0] = q_dot(g[0], wv);
        pw[1] = q_dot(g[1], wv);
        pw[2] = q_get(m_fma(g[2], wv, q_get(m_mul(g[2], wv), 1)), 0);
        const double JB = m_fma(d[0][2], pw[2], m_fma(d[0][0], pw[0], m_mul(d[0][1], pw[1])));
        const double JE = m_fma(d[1][2], pw[2], m_fma(d[1][0], pw[0], m_mul(d[1][1], pw[1])));
        const double w_gB = q_dot(wv, gB);
        const double wgb = m_mul(m_fma(-b, w_gB, JB), inv_B);
        const double t1 = q_cross(q_get(JE, c1), q_get(JE, c2), B1, Bq);
        const double t2 = q_cross(E1, Eq, q_get(JB, c1), q_get(JB, c2));
        const double wgv = m_fma(m_add(t1, t2), inv_B2, -m_mul(m_mul(m_mul(2.0, vE), w_gB), inv_B));
        double br = m_fma(mub * ph.inv_m * inv_g * inv_g, gB, m_mul(vpar, wgb));
        if constexpr (POT != POT_IDEAL) br = m_fma(ph.qm * vpar * Epar * ph.inv_c2 * inv_g, vE, br);
        br = m_add(br, wgv);
        const double bxbr = q_cross(q_get(b, c1), q_get(b, c2), q_get(br, c1), q_get(br, c2));
        F = m_fma(gamma * inv_B * ph.inv_qm, bxbr, wv);
        const double vw = q_dot(vE, wgb);
        Fu = m_fma(gamma, vw, POT == POT_IDEAL ? -mirror : m_fma(ph.qm, Epar, -mirror));
    }
    o.F = c == 3 ? Fu : F;
    o.vpar = vpar;
    o.Bm = Bm;
    o.b = b;
    o.r2 = r2;
    o.flags = flags;
    return o;
}

template <int POT>
__global__ void __launch_bounds__(32, 1) push_quad_kernel(const __grid_constant__ GridMeta<double> gm,
                                                       const __grid_constant__ Phys<double> ph,
                                                       const __grid_constant__ PushParams P)
{
    const int lane = threadIdx.x & 31, c = lane & 3;
    const unsigned quad = 0xFu << (lane & 28);
    const int64_t slot = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 2;
    // quads past the end shadow the last particle, so that whole warps shuffle
    const bool real = slot < P.st.n;
    const int64_t i = real ? slot : P.st.n - 1, cap = P.st.cap;
    const double dt = P.dt;
    double t0 = P.t0;
    int64_t step0 = P.step0;
    if (P.clock) {
        t0 = P.clock[0];
        step0 = (int64_t)P.clock[1] + P.kbase;
    }
    const StepW<double> w1 = {dt * 1.5, dt * -0.5, dt * (2.0 / 3.0), dt * (5.0 / 12.0), dt * (-1.0 / 12.0)};
    const uint32_t e = P.st.ens[i];
    // squared radii beyond which the shell's test is due, a rounding inside the shell
    const double r_in2 = P.ens[e].r_in > 0.0 ? P.ens[e].r_in * P.ens[e].r_in * (1.0 + 1e-14) : 0.0;
    const double r_out2 = P.ens[e].r_out > 0.0 ? P.ens[e].r_out * P.ens[e].r_out * (1.0 - 1e-14) : 0.0;
    double *const own = c == 0 ? P.st.x : (c == 1 ? P.st.y : (c == 2 ? P.st.z : P.st.u));
    double A = own[i], F0 = P.st.F0[c * cap + i], F1 = P.st.F1[c * cap + i];
    double S = P.st.s_rem[i], mub = P.st.mub[i], vpar0 = P.st.vpar[i], hprev = P.st.h_prev[i];
    double t_birth = P.st.t_birth[i], Bm0 = 0.0;
    uint32_t event = P.st.event[i], ncoll = P.st.ncoll[i], flags = P.st.flags[i];
    unsigned n_coll = 0, n_reb = 0;

    int next_tally = kNoTally;
    if (P.tally_on) {
        const int64_t K = P.tally.cadence;
        next_tally = (int)((K - 1 - (step0 % K)) % K);
    }
    int k = 0;
    do {
        const int k_end = min(P.n_steps, next_tally + 1);
        bool restart = false;
        // as in push_kernel: a restarting particle spends an iteration on its start-up history;
        // quads that are through evaluate on without effect until the warp's last is
        while (__any_sync(0xffffffffu, k < k_end)) {
            const bool act = k < k_end;
            const StepW<double> w = step_weights(w1, dt, hprev);
            const QuadEval a = quad_eval<POT, EV_PREDICTOR>(gm, ph, c, m_add(A, m_fma(w.a0, F0, m_mul(w.a1, F1))), mub, restart);
            if (act) {
                flags |= a.flags;
                if (restart) {
                    F0 = a.F;
                    vpar0 = a.vpar;
                    Bm0 = a.Bm;
                } else {
                    A += m_fma(w.c1, F1, m_fma(w.c0, F0, m_mul(w.cs, a.F)));
                }
            }
            const QuadEval o = quad_eval<POT, EV_CORRECTOR>(gm, ph, c, restart ? m_fma(-dt, F0, A) : A, mub, restart);
            if (!act) continue;
            flags |= o.flags;
            if (restart) {
                F1 = o.F;
                restart = false;
            } else {
                // Sect. 2.3: path length along B in this step
                const double ds = dt * (fabs(vpar0) + fabs(o.vpar)) * 0.5;
                bool collide = false;
                if (!P.no_scatter) {
                    if (P.collision_form == 0) {
                        S -= ds;
                        collide = S <= 0.0;
                    } else {
                        const uint4 wd = draw(P.st.id[i], P.seed, event++);
                        collide = u53(wd.x, wd.y) < 1.0 - exp(-ds / lambda_of(P, P.ens[e]));
                    }
                }
                auto at = [&](double v, int src) { return __shfl_sync(quad, v, src, 4); };
                bool reborn = false;
                if (!P.no_rebirth && (o.r2 < r_in2 || o.r2 > r_out2)) {
                    const double xx = at(A, 0), yy = at(A, 1), zz = at(A, 2);
                    const double r1 = sqrt(xx * xx + yy * yy + zz * zz);
                    reborn = r1 < P.ens[e].r_in || r1 > P.ens[e].r_out;
                }
                if (reborn || collide) {
                    RareState<double> s{at(A, 0), at(A, 1), at(A, 2), at(A, 3), S, mub, t_birth, event, ncoll};
                    s = rare_event<double>(P, ph, i, reborn, s, o.Bm, at(o.b, 0), at(o.b, 1), at(o.b, 2), t0,
                                           (long long)(P.kbase + k + 1));
                    A = c == 0 ? s.Rx : (c == 1 ? s.Ry : (c == 2 ? s.Rz : s.U));
                    S = s.S;
                    mub = s.mub;
                    t_birth = s.t_birth;
                    event = s.event;
                    ncoll = s.ncoll;
                    if (real && c == 0) {
                        if (reborn)
                            ++n_reb;
                        else
                            ++n_coll;
                    }
                    F0 = F1 = 0.0;
                    restart = true;
                    continue;
                }
                F1 = F0;
                F0 = o.F;
                vpar0 = o.vpar;
                Bm0 = o.Bm;
            }
            hprev = dt;
            ++k;
        }
        if (k == next_tally + 1) {
            next_tally = after_tally(next_tally, P.tally.cadence);
            const double x = q_get(A, 0), y = q_get(A, 1), z = q_get(A, 2), u = q_get(A, 3);
            const double t_new = step_time(t0, (long long)(P.kbase + k), P.dt);
            tally_sample<double>(P.tally, P, ph, e, x, y, z, u, mub, Bm0, t_new - t_birth, ncoll,
                                 real && c == 0 && t_birth >= P.tally.t_start && (int)e < P.tally.n_ens);
        }
    } while (k < P.n_steps);

    // what the last step leaves (see push_kernel); lanes of components x, u and x's F^n
    const unsigned bad = __ballot_sync(0xffffffffu, !m_finite(A) || (c == 0 && !m_finite(F0)));
    if ((bad >> (lane & 28)) & 9u) flags |= FLAG_NONFINITE;
    if (real) {
        own[i] = A;
        P.st.F0[c * cap + i] = F0;
        P.st.F1[c * cap + i] = F1;
        if (c == 0) {
            P.st.s_rem[i] = S;
            P.st.mub[i] = mub;
            P.st.vpar[i] = vpar0;
            P.st.h_prev[i] = hprev;
            P.st.t_birth[i] = t_birth;
            P.st.event[i] = event;
            P.st.ncoll[i] = ncoll;
            store_flags(P, i, flags);
        }
    }
    flush_counters(P, n_coll, n_reb);
}

// ----------------------------------------------------------------------------------------
// Injection (Sect. 3): site, mu0 and energy draws (Philox events 0 and 1), start-up history.
struct InjDraw {
    double mu0, pm; // pitch cosine and momentum magnitude |p| / m = gamma v
    uint4 w0;       // event 0 (mu0 and the first free path)
};

__device__ __forceinline__ InjDraw inj_draw(const EnsDev &E, uint32_t id, uint32_t seed, double m, double c2)
{
    InjDraw d;
    d.w0 = draw(id, seed, 0u);
    const uint4 w1 = draw(id, seed, 1u);
    d.mu0 = (E.mu_law == 1) ? 1.0 : u53(d.w0.x, d.w0.y);
    double Ek = E.E0;
    if (E.energy_law == 1) {
        const double a = 1.0 - E.E_index;
        const double uu = u53(w1.x, w1.y);
        Ek = pow(pow(E.E_lo, a) + uu * (pow(E.E_hi, a) - pow(E.E_lo, a)), 1.0 / a);
    }
    const double mc2 = m * c2;
    const double gam = 1.0 + Ek / mc2;
    d.pm = sqrt(c2) * sqrt(gam * gam - 1.0);
    return d;
}

template <typename T, bool TD, int POT>
__global__ void __launch_bounds__(256) inject_kernel(const GridMeta<T> gm, const Phys<T> ph,
                                                     const InjectParams P)
{
    const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= P.count)
        return;
    const int64_t i = P.slot0 + j;
    int e = 0;
    while (e + 1 < P.n_ens && j >= P.ens[e + 1].first - P.slot0)
        ++e;
    const EnsDev &E = P.ens[e];
    const uint32_t id = P.id0 + (uint32_t)j;
    const InjDraw d = inj_draw(E, id, P.seed, P.m, P.c2);
    const double mu0 = d.mu0, pm = d.pm;
    const uint4 w0 = d.w0;
    Sample<T> s;
    if constexpr (TD)
        gather_td<T, POT>(gm, (T)E.R0[0], (T)E.R0[1], (T)E.R0[2], (T)(P.t - gm.t_snap0), s);
    else
        gather<T, POT>(gm, (T)E.R0[0], (T)E.R0[1], (T)E.R0[2], s);
    const double Bm = (double)m_sqrt(dot3(s.B, s.B));
    const double u = mu0 * pm;
    const double mub = (1.0 - mu0 * mu0) * pm * pm * P.m / (2.0 * Bm);
    T F0[4], F1[4];
    Aux<T> a0x, a1x;
    const T x = (T)E.R0[0], y = (T)E.R0[1], z = (T)E.R0[2], uT = (T)u, mubT = (T)mub;
    const T dt = (T)P.dt_init;
    uint32_t flags = s.flags;
    const T t_inj = TD ? (T)(P.t - gm.t_snap0) : T(0);
    flags |= eval_F<T, TD, POT>(gm, ph, x, y, z, uT, mubT, F0, a0x, t_inj);
    flags |= eval_F<T, TD, POT>(gm, ph, x - dt * F0[0], y - dt * F0[1], z - dt * F0[2], uT - dt * F0[3],
                                mubT, F1, a1x, t_inj - dt);
    const int64_t cap = P.st.cap;
    P.st.x[i] = E.R0[0];
    P.st.y[i] = E.R0[1];
    P.st.z[i] = E.R0[2];
    P.st.u[i] = u;
    P.st.mub[i] = mub;
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        P.st.F0[c * cap + i] = (double)F0[c];
        P.st.F1[c * cap + i] = (double)F1[c];
    }
    P.st.vpar[i] = (double)a0x.vpar;
    P.st.s_rem[i] = -E.lambda * log(u53(w0.z, w0.w));
    P.st.h_prev[i] = P.dt_init;
    P.st.t_birth[i] = P.t;
    P.st.u_inj[i] = u;
    P.st.mub_inj[i] = mub;
    P.st.id[i] = id;
    P.st.ens[i] = (uint32_t)(P.ens_base + e);
    P.st.event[i] = 2u;
    P.st.ncoll[i] = 0u;
    P.st.flags[i] = flags;
    if (flags)
        atomicOr(P.gflags, flags);
}

// ----------------------------------------------------------------------------------------
// Split-step push (FP32 path): the step cut at its field evaluations, for sources that
// evaluate many points at once. Every particle walks the phases above at its own pace: a round
// consumes one field sample per unfinished particle and asks for the next one, so the two
// evaluations of a restart after a collision or rebirth are part of the rounds that the
// other particles' next step needs anyway, and a particle is behind by a step per event. After
// 2 n_steps rounds the few particles still behind go on in a compact list.
// (With PRED, CORR, POST and two restart kernels and four evaluations per step, in lockstep,
// 1024 particles took 97 us per step: each evaluation has a latency of about 16 us whatever the
// number of points.)
__device__ __forceinline__ void put_point(float *R, int64_t k, float x, float y, float z)
{
    R[3 * k] = x;
    R[3 * k + 1] = y;
    R[3 * k + 2] = z;
}

// one particle's progress: 4 x (steps done) + phase
__device__ __forceinline__ int32_t progress(int32_t step, int phase) { return 4 * step + phase; }

// store what phase 1 changed in a step without an event
__device__ __forceinline__ void store_step(const PushParams &P, int64_t i, const PState<float> &s)
{
    const int64_t cap = P.st.cap;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        P.st.F0[k * cap + i] = (double)s.F0[k];
        P.st.F1[k * cap + i] = (double)s.F1[k];
    }
    P.st.vpar[i] = (double)s.vpar0;
    P.st.s_rem[i] = AccOf<float>::to(s.S);
    P.st.h_prev[i] = (double)s.hprev;
    P.st.event[i] = s.event;
    store_flags(P, i, s.flags);
}

template <int KIND>
__global__ void __launch_bounds__(128) split_kernel(const __grid_constant__ Phys<float> ph, const __grid_constant__ SplitParams Q)
{
    using Acc = AccOf<float>;
    const PushParams &P = Q.P;
    const float dtT = (float)P.dt;
    const StepW<float> w1 = {dtT * 1.5f, dtT * -0.5f, dtT * (float)(2.0 / 3.0), dtT * (float)(5.0 / 12.0),
                             dtT * (float)(-1.0 / 12.0)};
    int64_t n = P.st.n;
    if (KIND == SPLIT_ROUND && Q.list_in) n = *Q.count_in;
    if (KIND == SPLIT_INJ_REQ || KIND == SPLIT_INJ_FIX || KIND == SPLIT_INJ_FIN) n = Q.n_new;
    unsigned n_coll = 0, n_reb = 0;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < n; k += stride) {
        if constexpr (KIND == SPLIT_INJ_REQ) {
            const EnsDev &E = P.ens[P.st.ens[Q.slot0 + k]];
            put_point(Q.req, k, (float)E.R0[0], (float)E.R0[1], (float)E.R0[2]);
            continue;
        }
        int64_t i = k;
        if (KIND == SPLIT_ROUND && Q.list_in) i = Q.list_in[k];
        if (KIND == SPLIT_INJ_FIX || KIND == SPLIT_INJ_FIN) i = Q.slot0 + k;
        int step = 0, phase = 0;
        if constexpr (KIND == SPLIT_ROUND) {
            const int32_t pr = Q.prog[i];
            step = pr >> 2;
            phase = pr & 3;
            if (step >= P.n_steps) continue;
        }
        PConst c;
        PState<float> s;
        load_particle(P, i, c, s);
        const StepW<float> w = step_weights(w1, dtT, s.hprev);
        Sample<float> smp;
        float Fo[4];
        Aux<float> ax;
        float px, py, pz, pu;
        int n_phase = 2;
        if constexpr (KIND == SPLIT_INIT) {
            phase_point(0, s, w, dtT, px, py, pz, pu);
            put_point(Q.req, i, px, py, pz);
            Q.prog[i] = progress(0, 0);
        } else if constexpr (KIND == SPLIT_ROUND) {
            load_sample(Q.S, k, Q.g_in_sample, smp);
            switch (sampled_phase(P, ph, Q.ideal, i, s, c, smp, w1, dtT, Q.kbase, step, phase, px, py, pz, n_coll, n_reb)) {
            case CHANGED_RU: store_RU(P, i, s); break;
            case CHANGED_STEP: store_step(P, i, s); break;
            case CHANGED_ALL: store_particle(P, i, s); break;
            case CHANGED_F0: store_F(P, i, s, 0); break;
            default: store_F(P, i, s, 1); break;
            }
            Q.prog[i] = progress(step, phase);
            if (step < P.n_steps) {
                int64_t slot = k;
                if (Q.list_out) {
                    slot = atomicAdd(Q.count_out, 1);
                    Q.list_out[slot] = (int32_t)i;
                }
                put_point(Q.req, slot, px, py, pz);
            }
        } else if constexpr (KIND == SPLIT_INJ_FIX) {
            // the injection's field-dependent part with this source: mu_B from |B| at the
            // site, F^n there, and the F^{n-1} request at X^n - dt F^n (Sect. 2.2)
            const InjDraw d = inj_draw(P.ens[c.e], P.st.id[i], P.seed, P.m, P.c2);
            load_sample(Q.S, k, Q.g_in_sample, smp);
            s.flags |= smp.flags;
            const double Bm = (double)m_sqrt(dot3(smp.B, smp.B));
            const double u = d.mu0 * d.pm;
            const double mub = (1.0 - d.mu0 * d.mu0) * d.pm * d.pm * P.m / (2.0 * Bm);
            s.U = Acc::from(u);
            s.mub = (float)mub;
            mub_lo_set<float>(mub, s.mub);
            rhs(smp, ph, Q.ideal, (float)u, (float)mub, Fo, ax);
            phase_consume(2, n_phase, i, s, c, Fo, ax, w, P, ph, dtT, P.t0, 0, n_coll, n_reb);
            phase_point(3, s, w, dtT, px, py, pz, pu);
            put_point(Q.req, k, px, py, pz);
            P.st.u[i] = u;
            P.st.mub[i] = mub;
            P.st.u_inj[i] = u;
            P.st.mub_inj[i] = mub;
            store_F(P, i, s, 0);
        } else if constexpr (KIND == SPLIT_INJ_FIN) {
            phase_point(3, s, w, dtT, px, py, pz, pu);
            load_sample(Q.S, k, Q.g_in_sample, smp);
            s.flags |= smp.flags;
            rhs(smp, ph, Q.ideal, pu, s.mub, Fo, ax);
            phase_consume(3, n_phase, i, s, c, Fo, ax, w, P, ph, dtT, P.t0, 0, n_coll, n_reb);
            if (!(m_finite(Acc::val(s.Rx)) && m_finite(Acc::val(s.U)) && m_finite(s.F0[0])))
                s.flags |= FLAG_NONFINITE;
            store_F(P, i, s, 1);
        }
    }
    if (KIND == SPLIT_ROUND) flush_counters(P, n_coll, n_reb);
}

// grid samples in the split-step layout (Sample fields, index-space derivatives with g)
__global__ void __launch_bounds__(128) grid_sample_kernel(const GridMeta<float> gm, const float *__restrict__ R,
                                                          int64_t cap, const int32_t *n_dev, float *__restrict__ S)
{
    int64_t n = cap;
    if (n_dev) n = *n_dev < cap ? *n_dev : cap;
    for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < n; k += (int64_t)gridDim.x * blockDim.x) {
        Sample<float> s;
        gather(gm, R[3 * k], R[3 * k + 1], R[3 * k + 2], s);
        float v[40];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            v[c] = s.B[c];
            v[3 + c] = s.E[c];
        }
#pragma unroll
        for (int d = 0; d < 3; ++d)
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                v[6 + 3 * d + c] = s.dB[d][c];
                v[15 + 3 * d + c] = s.dE[d][c];
                v[24 + 3 * d + c] = s.g[d][c];
            }
        v[33] = __uint_as_float(s.flags);
#pragma unroll
        for (int c = 0; c < 3; ++c)
            v[34 + c] = s.dPhi[c];
        v[37] = v[38] = v[39] = 0.f;
        float4 *q = reinterpret_cast<float4 *>(S + k * kSampleStride);
#pragma unroll
        for (int j = 0; j < 10; ++j)
            q[j] = make_float4(v[4 * j], v[4 * j + 1], v[4 * j + 2], v[4 * j + 3]);
    }
}

// ----------------------------------------------------------------------------------------
template <typename T>
static GridMeta<T> make_meta(const GridHost &g)
{
    GridMeta<T> m;
    m.nodes = static_cast<const T *>(g.nodes);
    m.n_r = g.n_r;
    m.n_th = g.n_th;
    m.n_ph = g.n_ph;
    m.ideal = g.ideal;
    m.r_min = (T)g.r_min;
    m.inv_dr = (T)(1.0 / g.dr);
    m.inv_dth = (T)(1.0 / g.dth);
    m.inv_dph = (T)(1.0 / g.dph);
    m.nodes1 = static_cast<const T *>(g.nodes1);
    m.span = g.nodes1 ? (T)(g.t_snap1 - g.t_snap0) : T(1);
    m.inv_span = g.nodes1 ? (T)(1.0 / (g.t_snap1 - g.t_snap0)) : T(0);
    m.t_snap0 = g.t_snap0;
    return m;
}

// The fused push and injection come in one variant per field mode: steady or time
// dependent (two snapshots), with or without the potential channel (two-fluid E_par).
template <typename T>
using PushFn = void (*)(const GridMeta<T>, const Phys<T>, const PushParams);
template <typename T>
using InjectFn = void (*)(const GridMeta<T>, const Phys<T>, const InjectParams);

// ideal: the grid's mode is 1 (E_par = 0), which has a variant of its own
template <typename T>
PushFn<T> push_fn(bool td, bool pot, bool ideal)
{
    if (td)
        return pot ? push_kernel<T, true, POT_ON> : (ideal ? push_kernel<T, true, POT_IDEAL> : push_kernel<T, true, POT_NONE>);
    return pot ? push_kernel<T, false, POT_ON> : (ideal ? push_kernel<T, false, POT_IDEAL> : push_kernel<T, false, POT_NONE>);
}

template <typename T>
InjectFn<T> inject_fn(bool td, bool pot)
{
    if (td)
        return pot ? inject_kernel<T, true, POT_ON> : inject_kernel<T, true, POT_NONE>;
    return pot ? inject_kernel<T, false, POT_ON> : inject_kernel<T, false, POT_NONE>;
}

// FP64, a steady field, and at most six warps of quads per SM (8.4 ms instead of 10.2; with
// eight 10.9)
bool push_quad_fits(int precision, const GridHost &g, int64_t n, int sms)
{
    return precision == 0 && !g.nodes1 && n > 0 && n <= (int64_t)sms * 48;
}

cudaError_t launch_push_quad(const GridHost &g, const PhysHost &ph, const PushParams &p, cudaStream_t s)
{
    cudaGetLastError(); // report this launch only
    const int grid = (int)((p.st.n + 7) / 8);
    const auto fn = g.ideal == 2 ? push_quad_kernel<POT_ON> : (g.ideal == 1 ? push_quad_kernel<POT_IDEAL> : push_quad_kernel<POT_NONE>);
    fn<<<grid, 32, 0, s>>>(make_meta<double>(g), make_phys<double>(ph), p);
    return cudaGetLastError();
}

static int push_threads(int precision, bool time_dependent)
{
    if (precision == 0) return time_dependent ? kPushThreads<double, true> : kPushThreads<double, false>;
    return time_dependent ? kPushThreads<float, true> : kPushThreads<float, false>;
}

int push_group(int precision) { return (int)(precision == 0 ? kSpread<double> : kSpread<float>); }

// One block per SM that holds all the threads the registers allow (FP32 of 934 000 particles
// 2.88e10 particle-steps/s with blocks of 128, 2.91e10 of 256, 2.99e10 of 512; two-fluid field and
// wind 2.14e10, 2.17e10, 2.25e10), or as many as the particles need: a block keeps its registers
// until its last thread is through, and what a small push does not use is there for another
// context's (four of 19 456 particles on their own streams, 20 000 steps: 96 ms in blocks of 512,
// 49 of 128; one alone 24 either way, and no size from 1000 to 160 000 takes longer).
int push_block(int precision, bool time_dependent, int64_t n, int sms)
{
    const int64_t per_sm = (n + sms - 1) / sms;
    return (int)std::max<int64_t>(128, std::min<int64_t>((per_sm + 127) / 128 * 128, push_threads(precision, time_dependent)));
}

void push_spread(PushParams &p, int block, int grid)
{
    const int64_t round = (int64_t)grid * block;
    p.spread_from = block % 128 == 0 ? p.st.n / round * round : INT64_MAX;
}

cudaError_t launch_push(int precision, const GridHost &g, const PhysHost &ph, const PushParams &p,
                        int block, int grid, cudaStream_t s)
{
    if (block < 1 || block > push_threads(precision, g.nodes1 != nullptr))
        return cudaErrorInvalidConfiguration;
    cudaGetLastError(); // report this launch only
    const bool td = g.nodes1 != nullptr, pot = g.ideal == 2, ideal = g.ideal == 1;
    if (precision == 0)
        push_fn<double>(td, pot, ideal)<<<grid, block, 0, s>>>(make_meta<double>(g), make_phys<double>(ph), p);
    else
        push_fn<float>(td, pot, ideal)<<<grid, block, 0, s>>>(make_meta<float>(g), make_phys<float>(ph), p);
    return cudaGetLastError();
}

cudaError_t launch_inject(int precision, const GridHost &g, const PhysHost &ph,
                          const InjectParams &p, cudaStream_t s)
{
    const int block = 128;
    const int grid = (int)((p.count + block - 1) / block);
    if (grid == 0)
        return cudaSuccess;
    const bool td = g.nodes1 != nullptr, pot = g.ideal == 2;
    if (precision == 0)
        inject_fn<double>(td, pot)<<<grid, block, 0, s>>>(make_meta<double>(g), make_phys<double>(ph), p);
    else
        inject_fn<float>(td, pot)<<<grid, block, 0, s>>>(make_meta<float>(g), make_phys<float>(ph), p);
    return cudaGetLastError();
}

cudaError_t launch_split(int kind, const PhysHost &ph, const SplitParams &p, int64_t n, cudaStream_t s)
{
    const Phys<float> q = make_phys<float>(ph);
    // one warp per block up to an SM's worth of warps each: a round of few particles is latency
    const int block = n <= 152 * 128 ? 32 : 128;
    int64_t blocks = (n + block - 1) / block;
    if (blocks > 152 * 64) blocks = 152 * 64;
    if (blocks < 1) blocks = 1;
    cudaGetLastError();
    switch (kind) {
    case SPLIT_INIT: split_kernel<SPLIT_INIT><<<(int)blocks, block, 0, s>>>(q, p); break;
    case SPLIT_ROUND: split_kernel<SPLIT_ROUND><<<(int)blocks, block, 0, s>>>(q, p); break;
    case SPLIT_INJ_REQ: split_kernel<SPLIT_INJ_REQ><<<(int)blocks, block, 0, s>>>(q, p); break;
    case SPLIT_INJ_FIX: split_kernel<SPLIT_INJ_FIX><<<(int)blocks, block, 0, s>>>(q, p); break;
    case SPLIT_INJ_FIN: split_kernel<SPLIT_INJ_FIN><<<(int)blocks, block, 0, s>>>(q, p); break;
    default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

cudaError_t launch_grid_samples(const GridHost &g, const float *R, int64_t cap, const int32_t *n_dev, float *S,
                                cudaStream_t s)
{
    int64_t blocks = (cap + 127) / 128;
    if (blocks > 152 * 64) blocks = 152 * 64;
    if (blocks < 1) blocks = 1;
    cudaGetLastError();
    grid_sample_kernel<<<(int)blocks, 128, 0, s>>>(make_meta<float>(g), R, cap, n_dev, S);
    return cudaGetLastError();
}

cudaError_t preload_kernels()
{
    cudaFuncAttributes a;
    cudaError_t e = cudaSuccess;
    for (int v = 0; v < 8 && e == cudaSuccess; ++v) {
        e = cudaFuncGetAttributes(&a, push_fn<float>(v & 1, v & 2, v & 4));
        if (e == cudaSuccess) e = cudaFuncGetAttributes(&a, push_fn<double>(v & 1, v & 2, v & 4));
    }
    if (e == cudaSuccess) e = cudaFuncGetAttributes(&a, push_quad_kernel<POT_ON>);
    if (e == cudaSuccess) e = cudaFuncGetAttributes(&a, push_quad_kernel<POT_IDEAL>);
    if (e == cudaSuccess) e = cudaFuncGetAttributes(&a, push_quad_kernel<POT_NONE>);
    return e;
}

int push_max_blocks_per_sm(int precision, int block, bool time_dependent, bool potential)
{
    int nb = 0;
    if (precision == 0)
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, push_fn<double>(time_dependent, potential, !potential), block, 0);
    else
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, push_fn<float>(time_dependent, potential, !potential), block, 0);
    return nb;
}

} // namespace gcp
