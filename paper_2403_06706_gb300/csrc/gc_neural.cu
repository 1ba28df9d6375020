// gc_neural.cu -- the neural field: parameters on the device, the training targets, the
// training's forward and backward passes, and Adam.
//
// Network and conventions (SIREN, Sitzmann et al. 2020): x = R / r_max; z1 = w0 (W1 x + b1),
// h_k = sin z_k, z_k = W_k h_{k-1} + b_k (k = 2..4), y = W5 h4 + b5. Outputs are the grid's
// eight channels scaled to O(1): B and |B| times (r / 1 AU)^2 / B_scale, E times
// (r / 1 AU) / E_scale, Phi / (E_scale 1 AU). The training minimises the mean squared error
// over samples and channels (Kingma & Ba 2015 for Adam) with the same arithmetic as the
// fused evaluation: W2..W5 and the activations h_1..h_4 in BF16, FP32 accumulation, FP32
// first layer and biases. The forward and backward passes are in gc_train.cu; the targets,
// Adam and the parameters' BF16 copies are here.
#include <algorithm>
#include <cmath>
#include <cstring>

#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include "gc_device.cuh"
#include "gc_neural.h"
#include "gc_siren.h"

namespace gcn {

using gcs::kSirenNParams;
using gcs::siren_oB;
using gcs::siren_oW;

namespace {

constexpr double kAU = 1.495978707e11;
constexpr double kPi = 3.14159265358979323846;

inline int blocks_for(int64_t n, int block, int cap = 152 * 16)
{
    const int64_t b = (n + block - 1) / block;
    return (int)(b < cap ? (b > 0 ? b : 1) : cap);
}

// BF16 copy of parameter i if it belongs to W2..W5
__device__ __forceinline__ void put_bf16(int64_t i, float p, __nv_bfloat16 *Wh, __nv_bfloat16 *W5p)
{
#pragma unroll
    for (int L = 2; L <= 4; ++L) {
        const int64_t o = siren_oW(L);
        if (i >= o && i < o + 65536) {
            Wh[(int64_t)(L - 2) * 65536 + (i - o)] = __float2bfloat16_rn(p);
            return;
        }
    }
    if (i >= siren_oW(5) && i < siren_oW(5) + 2048)
        W5p[i - siren_oW(5)] = __float2bfloat16_rn(p);
}

__global__ void k_to_bf16(const float *__restrict__ P, __nv_bfloat16 *Wh, __nv_bfloat16 *W5p)
{
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < kSirenNParams;
         i += (int64_t)gridDim.x * blockDim.x)
        put_bf16(i, P[i], Wh, W5p);
}

// Adam (Kingma & Ba 2015) with bias corrections bc1 = 1 - beta1^t, bc2 = 1 - beta2^t; clears G
__global__ void k_adam(float *__restrict__ P, float *__restrict__ G, float *__restrict__ M,
                       float *__restrict__ V, float lr, float b1, float b2, float eps, float bc1, float bc2,
                       __nv_bfloat16 *Wh, __nv_bfloat16 *W5p)
{
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < kSirenNParams;
         i += (int64_t)gridDim.x * blockDim.x) {
        const float g = G[i];
        G[i] = 0.f; // the next batch adds to it
        const float m = b1 * M[i] + (1.0f - b1) * g;
        const float v = b2 * V[i] + (1.0f - b2) * g * g;
        M[i] = m;
        V[i] = v;
        const float p = P[i] - lr * (m / bc1) / (sqrtf(v / bc2) + eps);
        P[i] = p;
        put_bf16(i, p, Wh, W5p);
    }
}

// The eight channels of the trilinear grid interpolant at x (scaled by r_max), scaled as the
// network's outputs. Same cell conventions as the push's gather: node-centred, poles
// included, periodic in phi, clamped to the edge cells.
struct TargetGeom {
    int n_r, n_th, n_ph;
    double r_min, dr, r_max, B_scale, E_scale;
};

template <typename T>
__device__ __forceinline__ void target_point(const T *__restrict__ nodes, const TargetGeom &g, float x, float y, float z,
                                             float *__restrict__ out)
{
    const double X = (double)x * g.r_max, Y = (double)y * g.r_max, Zc = (double)z * g.r_max;
    const double rho = sqrt(X * X + Y * Y), r = sqrt(X * X + Y * Y + Zc * Zc);
    const double th = atan2(rho, Zc);
    double ph = atan2(Y, X);
    if (ph < 0) ph += 2.0 * kPi;
    const double xr = (r - g.r_min) / g.dr, xt = th / (kPi / (g.n_th - 1)), xp = ph / (2.0 * kPi / g.n_ph);
    int i = (int)floor(xr);
    double fr = xr - i;
    if (i < 0) { i = 0; fr = 0; }
    else if (i > g.n_r - 2) { i = g.n_r - 2; fr = 1; }
    int j = (int)floor(xt);
    double ft = xt - j;
    if (j < 0) { j = 0; ft = 0; }
    else if (j > g.n_th - 2) { j = g.n_th - 2; ft = 1; }
    // a NaN (whose conversion is the lowest integer) reads the first cell and leaves a NaN in fp;
    // in r and theta the clamps above catch it
    int k = xp >= 0 ? (int)floor(xp) : 0;
    const double fp = xp - k;
    if (k >= g.n_ph) k -= g.n_ph;
    const int k1 = (k + 1 == g.n_ph) ? 0 : k + 1;
    double v[8] = {0, 0, 0, 0, 0, 0, 0, 0};
    for (int a = 0; a < 2; ++a)
        for (int b = 0; b < 2; ++b)
            for (int c = 0; c < 2; ++c) {
                const double w = (a ? fr : 1 - fr) * (b ? ft : 1 - ft) * (c ? fp : 1 - fp);
                const T *p = nodes + (((int64_t)(c ? k1 : k) * g.n_th + (j + b)) * g.n_r + (i + a)) * 8;
                for (int ch = 0; ch < 8; ++ch)
                    v[ch] += w * (double)p[ch];
            }
    const double a1 = r / kAU;
    const double sb = a1 * a1 / g.B_scale, se = a1 / g.E_scale;
    for (int ch = 0; ch < 3; ++ch) {
        out[ch] = (float)(v[ch] * sb);
        out[3 + ch] = (float)(v[3 + ch] * se);
    }
    out[6] = (float)(v[6] * sb);
    out[7] = (float)(v[7] / (g.E_scale * kAU));
}

template <typename T>
__global__ void k_targets(const T *__restrict__ nodes, const TargetGeom g, const float *__restrict__ x, int64_t n,
                          float *__restrict__ out)
{
    for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < n; q += (int64_t)gridDim.x * blockDim.x)
        target_point(nodes, g, x[3 * q], x[3 * q + 1], x[3 * q + 2], out + 8 * q);
}

// The same from an FP32 grid, in pairs of floats (value hi + lo, about 2^-45): GB300 runs
// FP64 at 1/64 of FP32, and a point takes some 500 FP64 operations and conversions above.
// Error-free sums and products (Dekker 1971, Knuth) carry every step below, so the result is
// the float nearest the FP64 one but for about one value in 10^5. 2^20 points of the 256 x 128
// x 256 grid: 688 us in FP64, 70 us so (the 8 corner records, at random, are 270 MB).
struct ff {
    float h, l;
};
__host__ __device__ inline ff ff_of(double d)
{
    const float h = (float)d;
    return {h, (float)(d - (double)h)};
}
__device__ __forceinline__ ff ff_norm(float h, float l) // |h| >= |l|
{
    const float s = __fadd_rn(h, l);
    return {s, __fsub_rn(l, __fsub_rn(s, h))};
}
__device__ __forceinline__ ff ff_sum(float a, float b) // a + b exactly
{
    const float s = __fadd_rn(a, b), t = __fsub_rn(s, a);
    return {s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, t)), __fsub_rn(b, t))};
}
__device__ __forceinline__ ff ff_prod(float a, float b) // a b exactly
{
    const float p = __fmul_rn(a, b);
    return {p, __fmaf_rn(a, b, -p)};
}
__device__ __forceinline__ ff ff_add(ff a, ff b)
{
    const ff s = ff_sum(a.h, b.h);
    return ff_norm(s.h, __fadd_rn(s.l, __fadd_rn(a.l, b.l)));
}
__device__ __forceinline__ ff ff_mul(ff a, ff b)
{
    const ff p = ff_prod(a.h, b.h);
    return ff_norm(p.h, __fmaf_rn(a.l, b.h, __fmaf_rn(a.h, b.l, p.l)));
}
__device__ __forceinline__ ff ff_mul(ff a, float b)
{
    const ff p = ff_prod(a.h, b);
    return ff_norm(p.h, __fmaf_rn(a.l, b, p.l));
}
// 1 / sqrt(a): one Newton step on the float estimate (relative error e < 2^-21 -> 3/8 e^2)
__device__ __forceinline__ ff ff_rsqrt(ff a)
{
    const float y = rsqrtf(a.h);
    const ff u = ff_mul(a, ff_prod(y, y));
    return ff_norm(y, __fmul_rn(__fmul_rn(0.5f, y), __fsub_rn(__fsub_rn(1.0f, u.h), u.l)));
}

// Index coordinate angle / step of the polar angle of (X, Y), given 1 / hypot(X, Y): the offset
// from the nearest of 256 tabulated angles by the arcsine's series, as in the push's FP64
// path (refine_angle); k256 = 2 pi / 256 / step, inv = 1 / step.
__device__ __forceinline__ ff ff_angle(ff X, ff Y, ff inv_h, const float4 *table, ff k256, ff inv)
{
    const int m = __float2int_rn(gcp::m_atan2(Y.h, X.h) * (float)kCircleInvStep) & (GC_CIRCLE_N - 1);
    const float4 cs = table[m];
    const ff yc = ff_mul(Y, ff{cs.x, cs.y}), xs = ff_mul(X, ff{cs.z, cs.w});
    const ff t = ff_mul(ff_add(yc, ff{-xs.h, -xs.l}), inv_h);
    const float t2 = t.h * t.h;
    const float p = fmaf(fmaf(t2, 5.0f / 112.0f, 3.0f / 40.0f), t2, 1.0f / 6.0f);
    const ff d = ff_norm(t.h, __fmaf_rn(t.h * t2, p, t.l));
    return ff_add(ff_mul(k256, (float)m), ff_mul(d, inv));
}

// cell index and fraction in [0, 1] of an index coordinate
__device__ __forceinline__ int ff_cell(ff x, ff &f)
{
    float fl = floorf(x.h);
    f = ff_norm(__fsub_rn(x.h, fl), x.l);
    if (f.h < 0.f) { // x.h whole, x.l negative
        fl -= 1.f;
        f = ff_norm(1.f, f.h);
    }
    return (int)fl;
}

struct TargetGeomF {
    ff rr, r0, kt, it, kp, ip; // r_max / dr, r_min / dr; 2 pi / 256 and 1 in units of the theta, phi steps
    ff au, ib, ie, ip7;        // r_max / AU, 1 / B_scale, 1 / E_scale, 1 / (E_scale AU)
};

__device__ __noinline__ void target_point_f64(const float *nodes, const TargetGeom &g, float x, float y, float z, float *out)
{
    target_point(nodes, g, x, y, z, out);
}

__global__ void __launch_bounds__(128) k_targets_ff(const float *__restrict__ nodes, const __grid_constant__ TargetGeom g,
                                                    const __grid_constant__ TargetGeomF G, const float *__restrict__ x,
                                                    int64_t n, float *__restrict__ out)
{
    __shared__ float4 table[GC_CIRCLE_N]; // cos and sin of the reference angles as pairs
    for (int m = threadIdx.x; m < GC_CIRCLE_N; m += blockDim.x) {
        const double2 cs = kUnitCircle[m];
        const ff c = ff_of(cs.x), s = ff_of(cs.y);
        table[m] = make_float4(c.h, c.l, s.h, s.l);
    }
    __syncthreads();
    for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < n; q += (int64_t)gridDim.x * blockDim.x) {
        const float X = x[3 * q], Y = x[3 * q + 1], Z = x[3 * q + 2];
        const ff rho2 = ff_add(ff_prod(X, X), ff_prod(Y, Y)), r2 = ff_add(rho2, ff_prod(Z, Z));
        float o[8];
        // pairs lose their low words near the limits of the format (and on the axis): FP64 there
        bool ok = rho2.h > 1e-20f && r2.h < 1e20f;
        if (ok) {
            const ff ir = ff_rsqrt(r2), irho = ff_rsqrt(rho2);
            const ff r = ff_mul(r2, ir), rho = ff_mul(rho2, irho);
            const ff b0 = ff_mul(r, G.rr);
            const ff xr = ff_add(b0, ff{-G.r0.h, -G.r0.l});
            const ff xt = ff_angle(ff{Z, 0.f}, rho, ir, table, G.kt, G.it);
            ff xp = ff_angle(ff{X, 0.f}, ff{Y, 0.f}, irho, table, G.kp, G.ip);
            if (xp.h < 0.f) xp = ff_add(xp, ff{(float)g.n_ph, 0.f});
            ff fr, ft, fp;
            int i = xr.h < -1.f ? -1 : (xr.h > (float)g.n_r ? g.n_r : ff_cell(xr, fr));
            int j = ff_cell(xt, ft), k = ff_cell(xp, fp);
            if (i < 0) { i = 0; fr = ff{0.f, 0.f}; }
            else if (i > g.n_r - 2) { i = g.n_r - 2; fr = ff{1.f, 0.f}; }
            if (j < 0) { j = 0; ft = ff{0.f, 0.f}; }
            else if (j > g.n_th - 2) { j = g.n_th - 2; ft = ff{1.f, 0.f}; }
            if (k >= g.n_ph) k -= g.n_ph;
            if (k < 0) k += g.n_ph;
            const int k1 = (k + 1 == g.n_ph) ? 0 : k + 1;
            const ff gr = ff_add(ff{1.f, 0.f}, ff{-fr.h, -fr.l}), gt = ff_add(ff{1.f, 0.f}, ff{-ft.h, -ft.l}),
                     gp = ff_add(ff{1.f, 0.f}, ff{-fp.h, -fp.l});
            float vh[8], vl[8];
#pragma unroll
            for (int ch = 0; ch < 8; ++ch)
                vh[ch] = vl[ch] = 0.f;
#pragma unroll
            for (int c = 0; c < 2; ++c)
#pragma unroll
                for (int b = 0; b < 2; ++b) {
                    const ff wtp = ff_mul(b ? ft : gt, c ? fp : gp);
                    const float4 *p = reinterpret_cast<const float4 *>(
                        nodes + (((int64_t)(c ? k1 : k) * g.n_th + (j + b)) * g.n_r + i) * 8);
#pragma unroll
                    for (int a = 0; a < 2; ++a) {
                        const ff w = ff_mul(a ? fr : gr, wtp);
                        const float4 pa = __ldg(p + 2 * a), pb = __ldg(p + 2 * a + 1);
                        const float pv[8] = {pa.x, pa.y, pa.z, pa.w, pb.x, pb.y, pb.z, pb.w};
#pragma unroll
                        for (int ch = 0; ch < 8; ++ch) {
                            const ff t = ff_prod(pv[ch], w.h);
                            const ff s = ff_sum(vh[ch], t.h);
                            vh[ch] = s.h;
                            vl[ch] = __fadd_rn(vl[ch], __fadd_rn(s.l, __fmaf_rn(pv[ch], w.l, t.l)));
                        }
                    }
                }
            const ff a1 = ff_mul(r, G.au);
            const ff sb = ff_mul(ff_mul(a1, a1), G.ib), se = ff_mul(a1, G.ie);
            ok = sb.h > 1e-20f && sb.h < 1e20f && se.h > 1e-20f && se.h < 1e20f && G.ip7.h > 1e-20f && G.ip7.h < 1e20f;
#pragma unroll
            for (int ch = 0; ch < 8; ++ch) {
                const float a = fabsf(vh[ch]);
                // zero, or in the range where the low words are normal (a NaN fails)
                ok = ok && (a == 0.f || (a > 1e-18f && a < 1e18f));
                const ff sc = ch < 3 || ch == 6 ? sb : (ch == 7 ? G.ip7 : se);
                const ff t = ff_prod(vh[ch], sc.h);
                o[ch] = __fadd_rn(t.h, __fmaf_rn(vl[ch], sc.h, __fmaf_rn(vh[ch], sc.l, t.l)));
            }
        }
        if (!ok) target_point_f64(nodes, g, X, Y, Z, o);
        float4 *dst = reinterpret_cast<float4 *>(out + 8 * q);
        if (((uintptr_t)out & 15u) == 0) {
            dst[0] = make_float4(o[0], o[1], o[2], o[3]);
            dst[1] = make_float4(o[4], o[5], o[6], o[7]);
        } else {
#pragma unroll
            for (int ch = 0; ch < 8; ++ch)
                out[8 * q + ch] = o[ch];
        }
    }
}

template <typename P>
cudaError_t dev_alloc(P **p, size_t bytes)
{
    return cudaMalloc((void **)p, bytes);
}

cudaError_t ensure_work(Neural &nn, int64_t rows)
{
    if (rows <= nn.wcap) return cudaSuccess;
    cudaFree(nn.act);
    nn.act = nullptr;
    nn.wcap = 0;
    cudaError_t e = dev_alloc(&nn.act, (size_t)6 * 256 * rows * sizeof(__nv_bfloat16));
    if (e == cudaSuccess) e = gcs::train_act_map(&nn.map_act, nn.act, rows);
    if (e == cudaSuccess) nn.wcap = rows;
    return e;
}

// forward and backward of one batch; adds sum r^2 to nn.d_loss and the gradient to grad
cudaError_t fwd_bwd(Neural &nn, const float *x, const float *t, int64_t n, float *grad, cudaStream_t s)
{
    const cudaError_t e = ensure_work(nn, n);
    return e != cudaSuccess ? e : gcs::train_fwd_bwd(nn.net, nn.map_act, x, t, n, grad, &nn.d_status->loss, s);
}

} // namespace

cudaError_t neural_free(Neural &nn)
{
    void *ptrs[] = {nn.P, nn.G, nn.Mo, nn.Vo, nn.Wh, nn.W5p, nn.act, nn.d_status, nn.Xs, nn.Ts};
    for (void *p : ptrs)
        if (p) cudaFree(p);
    if (nn.h_status) cudaFreeHost(nn.h_status);
    nn = Neural{};
    return cudaSuccess;
}

cudaError_t neural_set(Neural &nn, const float *params, bool on_device, double omega0, double r_max,
                       double B_scale, double E_scale, cudaStream_t s)
{
    cudaError_t e = cudaSuccess;
    const size_t pb = (size_t)kSirenNParams * sizeof(float);
    if (!nn.P) {
        e = dev_alloc(&nn.P, pb);
        if (e == cudaSuccess) e = dev_alloc(&nn.G, pb);
        if (e == cudaSuccess) e = dev_alloc(&nn.Mo, pb);
        if (e == cudaSuccess) e = dev_alloc(&nn.Vo, pb);
        if (e == cudaSuccess) e = dev_alloc(&nn.Wh, (size_t)3 * 65536 * sizeof(__nv_bfloat16));
        if (e == cudaSuccess) e = dev_alloc(&nn.W5p, (size_t)16 * 256 * sizeof(__nv_bfloat16));
        if (e == cudaSuccess) e = dev_alloc(&nn.d_status, sizeof(NeuralStatus));
        if (e == cudaSuccess) e = cudaMallocHost((void **)&nn.h_status, sizeof(NeuralStatus));
        if (e == cudaSuccess) e = cudaMemsetAsync(nn.d_status, 0, sizeof(NeuralStatus), s);
        if (e == cudaSuccess) e = cudaMemsetAsync(nn.W5p, 0, (size_t)16 * 256 * sizeof(__nv_bfloat16), s);
        if (e != cudaSuccess) {
            neural_free(nn);
            return e;
        }
        nn.net.P = nn.P;
        nn.net.Wh = nn.Wh;
        nn.net.W5p = nn.W5p;
        nn.net.err = &nn.d_status->err;
        e = gcs::siren_maps(nn.net);
        if (e != cudaSuccess) {
            neural_free(nn);
            return e;
        }
    }
    e = cudaMemcpyAsync(nn.P, params, pb, on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess) e = cudaMemsetAsync(nn.Mo, 0, pb, s);
    if (e == cudaSuccess) e = cudaMemsetAsync(nn.Vo, 0, pb, s);
    if (e != cudaSuccess) return e;
    k_to_bf16<<<blocks_for(kSirenNParams, 256), 256, 0, s>>>(nn.P, nn.Wh, nn.W5p);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    nn.omega0 = omega0;
    nn.net.omega0 = (float)omega0;
    nn.r_max = r_max;
    nn.B_scale = B_scale;
    nn.E_scale = E_scale;
    nn.adam_t = 0;
    nn.ready = true;
    return cudaSuccess;
}

cudaError_t neural_eval(Neural &nn, const float *x, int64_t n, float *y, float *J, cudaStream_t s)
{
    gcs::SirenIn in{x, n, nullptr, 1.0f, (float)nn.r_max};
    gcs::SirenOut o{};
    o.y = y;
    o.J = J;
    return gcs::siren_eval(nn.net, in, o, s);
}

cudaError_t neural_field(Neural &nn, const float *x, int64_t n, float *field, cudaStream_t s)
{
    gcs::SirenIn in{x, n, nullptr, 1.0f, (float)nn.r_max};
    gcs::SirenOut o{};
    o.field = field;
    o.field_stride = 24;
    o.B_scale = nn.B_scale;
    o.E_scale = nn.E_scale;
    return gcs::siren_eval(nn.net, in, o, s);
}

namespace {

// input and output of an evaluation at positions in m, with the physical field's scaling
void sample_io(const Neural &nn, const float *R, int64_t cap, const int32_t *n_dev, float *samples, int stride,
               gcs::SirenIn *in, gcs::SirenOut *o)
{
    *in = gcs::SirenIn{R, cap, n_dev, (float)(1.0 / nn.r_max), 1.0f};
    *o = gcs::SirenOut{};
    o->field = samples;
    o->field_stride = stride;
    o->B_scale = nn.B_scale;
    o->E_scale = nn.E_scale;
}

} // namespace

cudaError_t neural_field_at(Neural &nn, const float *R, int64_t cap, const int32_t *n_dev, float *samples,
                            int stride, cudaStream_t s)
{
    gcs::SirenIn in;
    gcs::SirenOut o;
    sample_io(nn, R, cap, n_dev, samples, stride, &in, &o);
    return gcs::siren_eval(nn.net, in, o, s);
}

cudaError_t neural_push(Neural &nn, const gcp::PhysHost &phys, const gcp::PushParams &push, int ideal, cudaStream_t s)
{
    gcs::SirenIn in;
    gcs::SirenOut o;
    sample_io(nn, nullptr, push.st.n, nullptr, nullptr, gcp::kSampleStride, &in, &o);
    return gcs::siren_push(nn.net, in, o, phys, push, ideal, s);
}

cudaError_t neural_targets(const Neural &nn, const GridRef &g, const float *x, int64_t n, float *out, cudaStream_t s)
{
    if (n <= 0) return cudaSuccess;
    const int b = blocks_for(n, 128);
    const TargetGeom t{g.n_r, g.n_th, g.n_ph, g.r_min, g.dr, nn.r_max, nn.B_scale, nn.E_scale};
    if (g.is_f64) {
        k_targets<double><<<b, 128, 0, s>>>((const double *)g.nodes, t, x, n, out);
    } else {
        const double it = (g.n_th - 1) / kPi, ip = g.n_ph / (2.0 * kPi);
        const TargetGeomF f{ff_of(nn.r_max / g.dr), ff_of(g.r_min / g.dr), ff_of(kCircleStep * it), ff_of(it),
                            ff_of(kCircleStep * ip), ff_of(ip), ff_of(nn.r_max / kAU), ff_of(1.0 / nn.B_scale),
                            ff_of(1.0 / nn.E_scale), ff_of(1.0 / (nn.E_scale * kAU))};
        k_targets_ff<<<b, 128, 0, s>>>((const float *)g.nodes, t, f, x, n, out);
    }
    return cudaGetLastError();
}

cudaError_t neural_loss_grad(Neural &nn, const float *x, const float *t, int64_t n, float *grad, cudaStream_t s)
{
    // train_dw_kernel adds groups of four floats: a gradient that is not aligned for them (a slice
    // of a caller's flat buffer) is summed in the network's own and copied out
    const bool direct = grad && ((uintptr_t)grad & 15u) == 0;
    float *g = direct ? grad : nn.G;
    const size_t bytes = (size_t)kSirenNParams * sizeof(float);
    cudaError_t e = cudaMemsetAsync(g, 0, bytes, s);
    if (e == cudaSuccess) e = cudaMemsetAsync(&nn.d_status->loss, 0, sizeof(double), s);
    if (e == cudaSuccess) e = fwd_bwd(nn, x, t, n, g, s);
    if (e == cudaSuccess && grad && !direct) e = cudaMemcpyAsync(grad, g, bytes, cudaMemcpyDeviceToDevice, s);
    return e;
}

cudaError_t neural_status_copy(Neural &nn, cudaStream_t s)
{
    return cudaMemcpyAsync(nn.h_status, nn.d_status, sizeof(NeuralStatus), cudaMemcpyDeviceToHost, s);
}

int neural_error(Neural &nn, cudaStream_t s)
{
    const int v = nn.h_status->err;
    if (v && cudaMemsetAsync(&nn.d_status->err, 0, sizeof(int), s) != cudaSuccess) return -1;
    return v;
}

cudaError_t neural_adam(Neural &nn, double lr, double beta1, double beta2, double eps, cudaStream_t s)
{
    ++nn.adam_t;
    const double bc1 = 1.0 - std::pow(beta1, (double)nn.adam_t), bc2 = 1.0 - std::pow(beta2, (double)nn.adam_t);
    k_adam<<<blocks_for(kSirenNParams, 256), 256, 0, s>>>(nn.P, nn.G, nn.Mo, nn.Vo, (float)lr, (float)beta1,
                                                         (float)beta2, (float)eps, (float)bc1, (float)bc2, nn.Wh,
                                                         nn.W5p);
    return cudaGetLastError();
}

cudaError_t neural_fit(Neural &nn, const GridRef &g, const float *samples, bool on_device, int64_t n_samples,
                       int64_t batch, int n_epochs, double lr, double beta1, double beta2, double eps,
                       float *loss_out, cudaStream_t s)
{
    cudaError_t e = cudaSuccess;
    if (n_samples > nn.scap) {
        cudaFree(nn.Xs);
        cudaFree(nn.Ts);
        nn.Xs = nullptr;
        nn.Ts = nullptr;
        nn.scap = 0;
        e = dev_alloc(&nn.Xs, (size_t)n_samples * 3 * sizeof(float));
        if (e == cudaSuccess) e = dev_alloc(&nn.Ts, (size_t)n_samples * 8 * sizeof(float));
        if (e != cudaSuccess) return e;
        nn.scap = n_samples;
    }
    e = cudaMemcpyAsync(nn.Xs, samples, (size_t)n_samples * 3 * sizeof(float),
                        on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess) e = neural_targets(nn, g, nn.Xs, n_samples, nn.Ts, s);
    if (e != cudaSuccess) return e;
    const int64_t nb = n_samples / batch;
    e = cudaMemsetAsync(nn.G, 0, (size_t)kSirenNParams * sizeof(float), s);
    for (int ep = 0; ep < n_epochs; ++ep) {
        if (e == cudaSuccess) e = cudaMemsetAsync(&nn.d_status->loss, 0, sizeof(double), s);
        for (int64_t b = 0; b < nb && e == cudaSuccess; ++b) {
            e = fwd_bwd(nn, nn.Xs + b * batch * 3, nn.Ts + b * batch * 8, batch, nn.G, s);
            if (e == cudaSuccess) e = neural_adam(nn, lr, beta1, beta2, eps, s);
        }
        if (e != cudaSuccess) return e;
        e = neural_status_copy(nn, s);
        if (e == cudaSuccess) e = cudaStreamSynchronize(s);
        if (e != cudaSuccess) return e;
        if (loss_out) loss_out[ep] = (float)(nn.h_status->loss / (double)(nb * batch * 8));
    }
    return cudaSuccess;
}

} // namespace gcn
