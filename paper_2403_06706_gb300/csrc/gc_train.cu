// gc_train.cu -- the training's forward and backward passes on the tensor cores (tcgen05,
// TMA, tensor memory): loss and gradient of the SIREN on one batch in two kernels.
//
// Kernel 1, siren_train_kernel: persistent, one CTA per SM, 64 samples per tile. A tile runs
// the whole chain without leaving the SM:
//   z1 = w0 (W1 x + b1), h_k = sin z_k, z_k = W_k h_{k-1} + b_k (k = 2..4), y = W5 h4 + b5,
//   dy = gscale (y - t), dz4 = (W5^T dy) cos z4, dz_{k-1} = (W_k^T dz_k) cos z_{k-1}.
// Products with W2..W4 and the output product run as D = W . H^T (M = 128 features, N = 64
// samples), so a thread owns one feature of each half: it adds the bias, takes sine and
// cosine of the accumulator, writes h (BF16) as the next layer's operand and puts the cosine
// (FP32) back into the accumulator's place in tensor memory, where the backward pass finds
// it: the pre-activations never go to memory. The three cosines and one D region fill the
// 512 columns (z1, three FMAs, is recomputed). Bias gradients, dW1 and dW5 accumulate in
// the owner's registers over all tiles of the launch.
// The BF16 activations h1..h3 and dz2..dz4 leave through TMA stores straight from the
// operand buffers, feature-major ([feature][sample]).
// Kernel 2, train_dw_kernel: dW_k = dZ_k H_{k-1}^T over the batch for the three layers in
// one launch, both operands K-major in that layout; the batch is split so that the CTAs of
// all layers fill the SMs once, and the splits add up by FP32 atomics.
//
// What bounds kernel 1: the tile is one dependent chain of 13 steps, about 56 000 cycles (203 us
// for the seven rounds of tiles of 65536 samples at 1.95 GHz). In it the CUDA cores issue 87 000
// warp instructions (sine and cosine of 4 x 256 pre-activations per sample, dW5), 21 700 slots of
// each scheduler, and the tensor cores take 10 000 cycles (a 128 x 64 x 16 MMA takes 48: shared
// memory). 203 us of 271 us for loss and gradient; kernel 2 takes 40 us, reading 300 MB, two
// thirds of them from memory. Before, each layer made passes over
// [sample][256] buffers (FP32 pre-activations, their gradients: 2 GB of traffic): 905 us.
// Warp roles of kernel 1 (608 threads): warps 0-15 compute (warp w: features 32 (w % 4) +
// lane of a half, samples 16 (w / 4) ..), warp 16 issues MMAs, warp 17 TMA loads of the
// weights (three 32 KB stages), warp 18 TMA stores. Every mbarrier wait is bounded
// and reports through the error word instead of hanging.
#include <type_traits>

#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include "gc_f32x2.cuh"
#include "gc_siren.h"
#include "gc_tc.cuh"

namespace gcs {

using namespace tc;

namespace {

constexpr int kRows = 64;                      // samples per tile
constexpr int kStagesW = 3;                    // weight ring depth
constexpr uint32_t kBoxBytes = 128u * 128u;    // one TMA box of weights: 128 rows x 64 bf16
constexpr uint32_t kStageBytes = 2 * kBoxBytes; // 128 x 128 weights
constexpr uint32_t kActBytes = 256u * 128u;    // 256 features x 64 samples bf16
constexpr uint32_t kW5Bytes = 4u * 16u * 128u; // W5 padded to 16 rows: 4 boxes of 16 x 64
// Samples of a batch up to which sine and cosine are the library's, one value at a time. The
// fast ones differ from them in the last place; where that moves a BF16 rounding, everything
// behind it in the sample is rounded anew, and the gradient moves by 8e-4 / sqrt(samples):
// 3.5e-5 for 512, 4e-6 for 32768 (either is 2e-3 from the gradient in FP64, BF16's rounding).
// So that small batches take the same roundings as plain sinf and cosf, and keep the results
// that they have always had: within 1.3e-6. That is what the line is for; it is neither the
// faster side (loss and gradient of 128, 4096, 8192, 16384 samples 70.5, 82, 94, 130 us here, 62,
// 70, 82, 107 with the fast ones; 215 at 512 and 395 at 16384 with a pass over memory per layer)
// nor the more accurate one (rms error of sine and cosine on |z| <= 30 1.9e-8 here, 1.7e-8 there).
constexpr int64_t kLibrarySines = 16384;
constexpr int kStagesPerTile = 24;             // 6 products x 4
constexpr int kComputeThreads = 512;
constexpr int kThreads = 608;
constexpr int kMmaWarp = 16, kTmaWarp = 17, kStoreWarp = 18;
// two activation buffers, W5 (its M = 128 descriptor reads on into the ring: rows past 8 of
// the output product are not used), ring, W5 in float, points, dy
constexpr size_t kOffW5 = 2 * kActBytes;
constexpr size_t kOffRing = kOffW5 + kW5Bytes;
constexpr size_t kOffW5f = kOffRing + kStagesW * kStageBytes;
constexpr size_t kOffPts = kOffW5f + 8 * 256 * 4;
constexpr size_t kOffDy = kOffPts + 16 * 16 * 16;
constexpr size_t kOffAW5 = kOffDy + kRows * 8 * 4;              // dW5 sums, [16][512 threads]
constexpr size_t kOffR = kOffAW5 + 16 * kComputeThreads * 4;  // residuals, [8][64]
constexpr size_t kOffBar = kOffR + kRows * 8 * 4;
constexpr size_t kSmemTrain = kOffBar + 256 + 1024;
static_assert(kSmemTrain <= 227 * 1024, "shared memory");

struct TrainParams {
    const float *P;              // master parameters
    const __nv_bfloat16 *W5p;    // W5 in BF16, 16 rows
    const float *x, *t;          // samples and targets
    int64_t n;                   // samples, a multiple of 64
    float omega0, gscale;
    float *G;                    // gradient (added to)
    double *loss;                // sum of squared residuals (added to)
    int *err;
};

// tensor-memory regions of 128 columns (64 samples x 2 halves)
__host__ __device__ constexpr uint32_t region(int r) { return (uint32_t)r * 128u; }

// 16 consecutive samples (16 rg ..) of one feature into an operand buffer; frow points at the
// feature's 128-byte row, swizzled by its row in the 8-row atom
__device__ __forceinline__ void store_rows16(uint8_t *frow, uint32_t rsw, int rg, const float (&o)[16])
{
#pragma unroll
    for (int c = 0; c < 2; ++c) {
        uint4 pk;
        pk.x = pack_bf16(o[8 * c], o[8 * c + 1]);
        pk.y = pack_bf16(o[8 * c + 2], o[8 * c + 3]);
        pk.z = pack_bf16(o[8 * c + 4], o[8 * c + 5]);
        pk.w = pack_bf16(o[8 * c + 6], o[8 * c + 7]);
        *reinterpret_cast<uint4 *>(frow + ((uint32_t)(2 * rg + c) ^ rsw) * 16u) = pk;
    }
}

__device__ __forceinline__ void load_rows16(const uint8_t *frow, uint32_t rsw, int rg, float (&o)[16])
{
#pragma unroll
    for (int c = 0; c < 2; ++c) {
        const uint4 pk = *reinterpret_cast<const uint4 *>(frow + ((uint32_t)(2 * rg + c) ^ rsw) * 16u);
        const uint32_t w[4] = {pk.x, pk.y, pk.z, pk.w};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            o[8 * c + 2 * i] = __uint_as_float(w[i] << 16);
            o[8 * c + 2 * i + 1] = __uint_as_float(w[i] & 0xFFFF0000u);
        }
    }
}

// Sine and / or cosine of 16 values (in place where an output is the input). With LIB, and
// beyond the fast reduction's range, the library's, one value at a time and out of line:
// pre-activations of a trained network stay below about 10^2.
__device__ __noinline__ float2 sincos_any(float z)
{
    float s, c;
    sincosf(z, &s, &c);
    return make_float2(s, c);
}

template <bool LIB, bool SIN, bool COS>
__device__ __forceinline__ void sincos16(const float (&z)[16], float (&sn)[16], float (&cs)[16])
{
    float m = 0.f;
#pragma unroll
    for (int i = 0; i < 16; ++i)
        m = fmaxf(m, fabsf(z[i]));
    if (!LIB && m <= gcp::kSincosMax) {
#pragma unroll
        for (int i = 0; i < 16; i += 2) {
            float s[2], c[2];
            gcp::sincos2(gcp::p2_pack(z[i], z[i + 1]), s, c);
            if (SIN) { sn[i] = s[0]; sn[i + 1] = s[1]; }
            if (COS) { cs[i] = c[0]; cs[i + 1] = c[1]; }
        }
    } else {
#pragma unroll
        for (int i = 0; i < 16; ++i) {
            const float2 v = sincos_any(z[i]);
            if (SIN) sn[i] = v.x;
            if (COS) cs[i] = v.y;
        }
    }
}

template <bool LIB>
__global__ void __launch_bounds__(kThreads, 1)
    siren_train_kernel(const __grid_constant__ CUtensorMap mwh, const __grid_constant__ CUtensorMap mw5, const __grid_constant__ CUtensorMap mact,
                       const __grid_constant__ TrainParams p)
{
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    uint8_t *sAct[2] = {smem, smem + kActBytes};
    uint8_t *sW5 = smem + kOffW5;
    uint8_t *sW = smem + kOffRing;
    float *sW5f = (float *)(smem + kOffW5f);    // [8][256]
    float4 *sPts = (float4 *)(smem + kOffPts);  // [16 compute warps][16 samples]
    float *sDy = (float *)(smem + kOffDy);      // [8][64]
    float *sRes = (float *)(smem + kOffR);      // [8][64]
    float *sAW5 = (float *)(smem + kOffAW5) + threadIdx.x;
    uint64_t *full = (uint64_t *)(smem + kOffBar);
    uint64_t *empty = full + kStagesW;
    uint64_t *h_ready = empty + kStagesW; // [2]: a half of the operand written
    uint64_t *acc = h_ready + 2;          // [2]: accumulator of a half complete
    uint64_t *acc_out = acc + 2;          // output product complete
    uint64_t *st_read = acc_out + 1;      // the TMA store of the last operand has read it
    uint64_t *dy_ready = st_read + 1;     // [4]: dy of a row group written
    uint64_t *fin = dy_ready + 4;
    uint64_t *w5full = fin + 1;
    uint32_t *tmem_slot = (uint32_t *)(w5full + 1);
    volatile int *abort = (volatile int *)(tmem_slot + 1);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t n_tiles = p.n / kRows;

    if (threadIdx.x == 0) {
        for (int s = 0; s < kStagesW; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        for (int h = 0; h < 2; ++h) {
            mbar_init(&h_ready[h], kComputeThreads / 32);
            mbar_init(&acc[h], 1);
        }
        for (int r = 0; r < 4; ++r)
            mbar_init(&dy_ready[r], 32);
        mbar_init(st_read, 1);
        mbar_init(acc_out, 1);
        mbar_init(fin, 1);
        mbar_init(w5full, 1);
        *abort = 0;
        mbar_fence_init();
    }
    for (int i = threadIdx.x; i < 8 * 256; i += kThreads)
        sW5f[i] = __bfloat162float(p.W5p[i]);
    if (warp == kMmaWarp) {
        tmem_alloc(tmem_slot, 512);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;

    if (warp == kTmaWarp) {
        // ------------------------------------------------------------ TMA loads (weights)
        if (lane == 0) {
            uint32_t st = 0, par = 1, filled = 0;
            bool ok = true;
            mbar_expect_tx(w5full, kW5Bytes);
            for (int kb = 0; kb < 4; ++kb)
                tma_load_2d(sW5 + kb * 2048, &mw5, kb * 64, 0, w5full);
            for (int64_t t = blockIdx.x; t < n_tiles && ok; t += gridDim.x) {
#pragma unroll 1
                for (int c = 0; c < kStagesPerTile; ++c) {
                    if (!wait_abort(&empty[st], par, abort, p.err, 31)) {
                        ok = false;
                        break;
                    }
                    // product c / 4 (W2, W3, W4, then W4^T, W3^T, W2^T), stages in the MMA order:
                    // output half h, operand features 128 kh ..; the same boxes of 128 rows x 64
                    // columns serve both directions
                    const int pr = c >> 2, h = c & 1, kh = (c >> 1) & 1;
                    const int x = pr < 3 ? kh * 128 : h * 128, y = pr < 3 ? pr * 256 + h * 128 : (5 - pr) * 256 + kh * 128;
                    uint8_t *dst = sW + st * kStageBytes;
                    mbar_expect_tx(&full[st], kStageBytes);
                    tma_load_2d(dst, &mwh, x, y, &full[st]);
                    tma_load_2d(dst + kBoxBytes, &mwh, x + 64, y, &full[st]);
                    filled |= 1u << st;
                    if (++st == kStagesW) {
                        st = 0;
                        par ^= 1u;
                    }
                }
            }
            // the copies still in flight land before the CTA's shared memory is released: the
            // last copy of a stage behind st is of the running phase, of one from st on of the
            // phase before
            for (int j = 0; j < kStagesW; ++j)
                if (filled >> j & 1)
                    mbar_wait(&full[j], (uint32_t)j < st ? par ^ 1u : par);
            mbar_wait(w5full, 0);
        }
    } else if (warp == kMmaWarp) {
        // ------------------------------------------------------------ MMA issuer
        // The whole warp runs the loop and one elected lane issues. Descriptors are a constant
        // high word and a running low word: built from addresses per MMA, with the stage by a
        // division, four MMAs took 530 to 950 cycles to issue beside the compute warps of the
        // same scheduler, two to four times what the tensor cores need for them.
        {
            constexpr uint32_t id_fwd = idesc_bf16_f32(128, kRows, 0, 1), id_bwd = idesc_bf16_f32(128, kRows, 1, 1);
            const bool leader = elect_one();
            const uint32_t tm = __shfl_sync(0xffffffffu, tmem, 0);
            const uint32_t act_lo = desc_lo(smem_u32(sAct[0]), 1024); // buffer B: + kActBytes / 16
            const uint32_t w_lo = smem_u32(sW) >> 4;
            uint32_t st = 0, par = 0, nh = 0; // ring stage and its phase; operands
            bool ok = true;
            auto wait = [&](uint64_t *bar, uint32_t phase, int code) {
                const bool r = __all_sync(0xffffffffu, wait_abort(bar, phase & 1u, abort, p.err, code)) != 0;
                tc_fence_after();
                return r;
            };
            // one product: 4 stages of 8 MMAs, (output half, operand half) = (0, 0) (1, 0) (0, 1)
            // (1, 1); d its accumulator, b_lo its operand
            auto product = [&](auto bwd_tag, uint32_t d, uint32_t b_lo) {
                constexpr bool bwd = decltype(bwd_tag)::value;
#pragma unroll 1
                for (int q = 0; q < 4; ++q) {
                    const int h = q & 1, kh = q >> 1;
                    if (h == 0 && !wait(&h_ready[kh], nh, 32 + kh)) return false;
                    if (!wait(&full[st], par, 34)) return false;
                    if (leader) {
                        // forward: K-major, 64 operand features a box; backward: MN-major, 64
                        // output features a box
                        const uint32_t a_lo = w_lo + st * (kStageBytes / 16) + (bwd ? (kBoxBytes / 16) << 16 : 1u << 16);
                        const uint32_t bh = b_lo + kh * (8 * 2048 / 16), dh = d + h * 64;
#pragma unroll
                        for (int k = 0; k < 8; ++k) {
                            const uint32_t ao = bwd ? k * 2048 : (k >> 2) * kBoxBytes + (k & 3) * 32;
                            mma_bf16(dh, desc_of(desc_hi(1024), a_lo + ao / 16),
                                     desc_of(desc_hi(1024), bh + k * (2048 / 16)), bwd ? id_bwd : id_fwd, (uint32_t)(kh | k));
                        }
                        mma_commit(&empty[st]);
                        if (kh) mma_commit(&acc[h]);
                    }
                    __syncwarp();
                    if (++st == kStagesW) {
                        st = 0;
                        par ^= 1u;
                    }
                }
                ++nh;
                return true;
            };
            if (!wait(w5full, 0, 35)) ok = false;
            const uint32_t lo_a = act_lo, lo_b = act_lo + kActBytes / 16;
            for (int64_t t = blockIdx.x; t < n_tiles && ok; t += gridDim.x) {
                // forward: h1 (A) -> region 1, h2 (B) -> 2, h3 (A) -> 3, kept as cosines
#pragma unroll 1
                for (int k = 0; k < 3 && ok; ++k)
                    ok = product(std::false_type{}, tm + region(1) * (k + 1), k & 1 ? lo_b : lo_a);
                if (!ok) break;
                // output product y = W5 h4 (B) into region 0
                for (int kh = 0; kh < 2 && ok; ++kh) {
                    if (!wait(&h_ready[kh], nh, 32 + kh)) { ok = false; break; }
                    if (leader) {
                        const uint32_t w5_lo = desc_lo(smem_u32(sW5), 16);
#pragma unroll
                        for (int k8 = 0; k8 < 8; ++k8) {
                            const int k16 = kh * 8 + k8;
                            mma_bf16(tm + region(0), desc_of(desc_hi(1024), w5_lo + (k16 >> 2) * 128 + (k16 & 3) * 2),
                                     desc_of(desc_hi(1024), lo_b + k16 * 128), id_fwd, k16 ? 1u : 0u);
                        }
                        if (kh) mma_commit(acc_out);
                    }
                    __syncwarp();
                }
                if (!ok) break;
                ++nh;
                // backward: dz4 (A) -> region 0, dz3 (B) -> 3, dz2 (A) -> 0
#pragma unroll 1
                for (int k = 0; k < 3 && ok; ++k)
                    ok = product(std::true_type{}, tm + (k & 1 ? region(3) : region(0)), k & 1 ? lo_b : lo_a);
            }
            // all MMAs of this CTA complete before its tensor memory is released
            if (leader) {
                mma_commit(fin);
                mbar_wait(fin, 0);
            }
            __syncwarp();
        }
    } else if (warp == kStoreWarp) {
        // ------------------------------------------------------------ TMA stores
        if (lane == 0) {
            uint32_t nh = 0;
            bool ok = true;
            for (int64_t t = blockIdx.x; t < n_tiles && ok; t += gridDim.x) {
                // operands in order: h1 A, h2 B, h3 A, h4 B (not stored), dz4 A, dz3 B, dz2 A;
                // the next one is written only after this warp is through with the last
                for (int k = 0; k < 7 && ok; ++k) {
                    for (int h = 0; h < 2; ++h) {
                        if (!wait_abort(&h_ready[h], nh & 1u, abort, p.err, 36)) { ok = false; break; }
                        if (k == 3) continue;
                        const int slab = k < 3 ? k : 9 - k; // h1 h2 h3 -> 0 1 2, dz4 dz3 dz2 -> 5 4 3
                        tma_store_2d(&mact, (int)(t * kRows), slab * 256 + h * 128, sAct[k & 1] + h * (kActBytes / 2));
                        bulk_commit();
                    }
                    ++nh;
                    bulk_wait_read();
                    if (ok) mbar_arrive(st_read);
                }
            }
            bulk_wait_all();
        }
    } else {
        // ------------------------------------------------------------ compute warps
        const int lq = warp & 3, rg = warp >> 2;
        const float w0 = p.omega0;
        const int f0 = lq * 32 + lane; // feature of half 0 (half 1: + 128)
        const uint32_t lane_base = tmem + ((uint32_t)(lq * 32) << 16) + (uint32_t)(rg * 16);
        const uint32_t rsw = (uint32_t)(lane & 7);
        const uint32_t frow = (uint32_t)(f0 >> 3) * 1024u + rsw * 128u; // half 1: + 16 KB
        float4 *wpts = sPts + warp * 16;
        float aB[3][2], aB1[2], aW1[2][3], aB5 = 0.f;
        for (int o = 0; o < 16; ++o)
            sAW5[o * kComputeThreads] = 0.f;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            aB1[h] = 0.f;
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                aB[k][h] = 0.f;
                aW1[h][k] = 0.f;
            }
        }
        double ls = 0.0;
        const float b5 = p.P[siren_oB(5) + (lane & 7)];
        uint32_t na = 0, no = 0, ns = 0; // completed products (both halves), tiles, operands
        bool ok = true;
        // waits agree over the warp, so that it leaves together when one runs out
        auto wait = [&](uint64_t *bar, uint32_t phase, int code) {
            return __all_sync(0xffffffffu, wait_abort(bar, phase & 1u, abort, p.err, code)) != 0;
        };
        auto wait_acc = [&](int h) {
            if (!wait(&acc[h], na, 37)) return false;
            na += h;
            tc_fence_after();
            return true;
        };
        // the TMA store of the operand written last has read it
        auto wait_store = [&]() { return wait(st_read, ns++, 38); };
        auto announce = [&](int h) {
            fence_proxy_async_smem();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&h_ready[h]);
        };
        for (int64_t t = blockIdx.x; t < n_tiles && ok; t += gridDim.x) {
            const bool first = t == blockIdx.x;
            const int64_t row0 = t * kRows + rg * 16;
            __syncwarp();
            if (lane < 16) {
                const float *xp = p.x + 3 * (row0 + lane);
                wpts[lane] = make_float4(__ldg(xp), __ldg(xp + 1), __ldg(xp + 2), 0.f);
            }
            __syncwarp();
            // ---- layer 1 (CUDA cores)
            if (!first && !wait_store()) break;
#pragma unroll 1
            for (int h = 0; h < 2; ++h) {
                const int f = f0 + h * 128;
                const float wa = __ldg(p.P + siren_oW(1) + 3 * f), wb = __ldg(p.P + siren_oW(1) + 3 * f + 1),
                            wc = __ldg(p.P + siren_oW(1) + 3 * f + 2), b1 = __ldg(p.P + siren_oB(1) + f);
                float v[16], o[16];
#pragma unroll
                for (int i = 0; i < 16; ++i) {
                    const float4 q = wpts[i];
                    v[i] = w0 * fmaf(wa, q.x, fmaf(wb, q.y, fmaf(wc, q.z, b1)));
                }
                sincos16<LIB, true, false>(v, o, v);
                store_rows16(sAct[0] + frow + h * (kActBytes / 2), rsw, rg, o);
                announce(h);
            }
            // ---- layers 2-4: h_k -> operand, cos z_k -> tensor memory
#pragma unroll 1
            for (int k = 0; k < 3 && ok; ++k) {
                const int buf = (k & 1) ^ 1;
                if (!wait_store()) { ok = false; break; }
#pragma unroll 1
                for (int h = 0; h < 2; ++h) {
                    const float b = __ldg(p.P + siren_oB(k + 2) + f0 + h * 128);
                    if (!wait_acc(h)) { ok = false; break; }
                    const uint32_t ta = lane_base + region(k + 1) + h * 64;
                    float v[16], o[16];
                    tmem_ld16(ta, v);
#pragma unroll
                    for (int i = 0; i < 16; ++i)
                        v[i] += b;
                    float c[16];
                    sincos16<LIB, true, true>(v, o, c);
                    store_rows16(sAct[buf] + frow + h * (kActBytes / 2), rsw, rg, o);
                    tmem_st16(ta, c);
                    announce(h);
                }
            }
            if (!ok) break;
            // ---- output residuals: dy = gscale (y - t) of this row group, in its warp lq = 0
            if (lq == 0) {
                float tt[16];
                if (lane < 8)
#pragma unroll
                    for (int i = 0; i < 16; ++i)
                        tt[i] = __ldg(p.t + (row0 + i) * 8 + lane);
                if (!wait(acc_out, no, 39)) break;
                tc_fence_after();
                float v[16];
                tmem_ld16(lane_base + region(0), v);
                if (lane < 8)
#pragma unroll
                    for (int i = 0; i < 16; ++i) {
                        const float r = v[i] + b5 - tt[i];
                        const float dy = p.gscale * r;
                        aB5 += dy;
                        sRes[lane * kRows + rg * 16 + i] = r;
                        sDy[lane * kRows + rg * 16 + i] = dy;
                    }
                tc_fence_before();
                mbar_arrive(&dy_ready[rg]);
            }
            if (!wait(&dy_ready[rg], no, 40)) break;
            ++no;
            {
                // the loss, in FP64 (1/64 rate): one residual per lane of the row group's warps
                const double r = (double)sRes[(lq * 2 + (lane >> 4)) * kRows + rg * 16 + (lane & 15)];
                ls += r * r;
            }
            // ---- dz4 (and dW5) -> operand A
            if (!wait_store()) break;
#pragma unroll 1
            for (int h = 0; h < 2; ++h) {
                float v[16], hv[16];
                load_rows16(sAct[1] + frow + h * (kActBytes / 2), rsw, rg, hv);
                unsigned long long dh[8];
#pragma unroll
                for (int o = 0; o < 8; ++o) {
                    const unsigned long long w5 = gcp::p2_bcast(sW5f[o * 256 + f0 + h * 128]);
                    unsigned long long a = 0;
#pragma unroll
                    for (int i = 0; i < 4; ++i) { // four samples at a time
                        const ulonglong2 dy =
                            *reinterpret_cast<const ulonglong2 *>(sDy + o * kRows + rg * 16 + 4 * i);
                        const unsigned long long ha = gcp::p2_pack(hv[4 * i], hv[4 * i + 1]),
                                                 hb = gcp::p2_pack(hv[4 * i + 2], hv[4 * i + 3]);
                        dh[2 * i] = o ? gcp::p2_fma(dy.x, w5, dh[2 * i]) : gcp::p2_mul(dy.x, w5);
                        dh[2 * i + 1] = o ? gcp::p2_fma(dy.y, w5, dh[2 * i + 1]) : gcp::p2_mul(dy.y, w5);
                        a = gcp::p2_fma(dy.x, ha, a);
                        a = gcp::p2_fma(dy.y, hb, a);
                    }
                    float a0, a1;
                    gcp::p2_split(a, a0, a1);
                    sAW5[(h * 8 + o) * kComputeThreads] += a0 + a1;
                }
                float s = 0.f;
                tmem_ld16(lane_base + region(3) + h * 64, v);
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    float d0, d1;
                    gcp::p2_split(dh[i], d0, d1);
                    v[2 * i] *= d0;
                    v[2 * i + 1] *= d1;
                    s += v[2 * i];
                    s += v[2 * i + 1];
                }
                if (h == 0)
                    aB[2][0] += s;
                else
                    aB[2][1] += s;
                store_rows16(sAct[0] + frow + h * (kActBytes / 2), rsw, rg, v);
                announce(h);
            }
            // ---- dz3 -> operand B (D in region 0, cosine in 2), dz2 -> operand A (3, 1)
#pragma unroll
            for (int k = 1; k >= 0; --k) {
                if (ok && !wait_store()) ok = false;
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    if (!ok || !wait_acc(h)) { ok = false; break; }
                    float v[16], c[16];
                    tmem_ld16(lane_base + (k ? region(0) : region(3)) + h * 64, v);
                    tmem_ld16(lane_base + region(k + 1) + h * 64, c);
                    float s = 0.f;
#pragma unroll
                    for (int i = 0; i < 16; ++i) {
                        v[i] *= c[i];
                        s += v[i];
                    }
                    aB[k][h] += s;
                    store_rows16(sAct[k] + frow + h * (kActBytes / 2), rsw, rg, v);
                    announce(h);
                }
            }
            // ---- dz1: dW1, db1 (D in region 0, z1 recomputed)
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                if (!ok) break;
                const int f = f0 + h * 128;
                const float wa = __ldg(p.P + siren_oW(1) + 3 * f), wb = __ldg(p.P + siren_oW(1) + 3 * f + 1),
                            wc = __ldg(p.P + siren_oW(1) + 3 * f + 2), b1 = __ldg(p.P + siren_oB(1) + f);
                float v[16], c[16];
#pragma unroll
                for (int i = 0; i < 16; ++i) {
                    const float4 q = wpts[i];
                    c[i] = w0 * fmaf(wa, q.x, fmaf(wb, q.y, fmaf(wc, q.z, b1)));
                }
                sincos16<LIB, false, true>(c, v, c);
                if (!wait_acc(h)) { ok = false; break; }
                tmem_ld16(lane_base + region(0) + h * 64, v);
#pragma unroll
                for (int i = 0; i < 16; ++i) {
                    const float4 q = wpts[i];
                    const float d = v[i] * c[i] * w0;
                    aB1[h] += d;
                    aW1[h][0] = fmaf(d, q.x, aW1[h][0]);
                    aW1[h][1] = fmaf(d, q.y, aW1[h][1]);
                    aW1[h][2] = fmaf(d, q.z, aW1[h][2]);
                }
            }
        }
        // this thread's sums over the launch
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int f = f0 + h * 128;
#pragma unroll
            for (int o = 0; o < 8; ++o)
                atomicAdd(p.G + siren_oW(5) + o * 256 + f, sAW5[(h * 8 + o) * kComputeThreads]);
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                atomicAdd(p.G + siren_oB(k + 2) + f, aB[k][h]);
                atomicAdd(p.G + siren_oW(1) + 3 * f + k, aW1[h][k]);
            }
            atomicAdd(p.G + siren_oB(1) + f, aB1[h]);
        }
        if (lq == 0 && lane < 8)
            atomicAdd(p.G + siren_oB(5) + lane, aB5);
        for (int off = 16; off > 0; off >>= 1)
            ls += __shfl_down_sync(0xffffffffu, ls, off);
        if (lane == 0)
            atomicAdd(p.loss, ls);
    }
    tc_fence_before();
    __syncthreads();
    if (warp == kMmaWarp) {
        tc_fence_after();
        tmem_dealloc(tmem, 512);
    }
}

// ----------------------------------------------------------------------------------------
// dW_k = dZ_k H_{k-1}^T: one CTA computes 128 output features (blockIdx.y) x 256 inputs of
// one layer (blockIdx.z) over a split of the batch (blockIdx.x), 64 samples per stage.
// The sums in tensor memory are rounded towards zero and lose up to 1e-7 of the gradient per
// stage where the samples' terms have one sign, so they are kept short: kDwChunk stages go into
// one accumulator, and while the next chunk's MMAs fill the other (2 x 256 columns), eight warps
// add it to FP32 sums in registers, rounded to nearest. 2^22 samples against
// the mean of eight parts: 2.3e-7 (2.6e-4 with one such sum per split of the batch). The drains
// hide behind the operands' copies, which bound the kernel (one batch of a fit, 8192 and 65536
// samples: 89.3 and 264.5 us, as with one sum per split), once the sums leave by whole rows:
// added to the gradient straight from the registers, in sectors of 32 rows, 91.4 and 266.8.
constexpr int kDwStages = 4;
constexpr int kDwChunk = 2;
constexpr int kDwSumWarps = 8, kDwThreads = 32 * (kDwSumWarps + 1); // the last warp issues
constexpr uint32_t kDwStageBytes = (128u + 256u) * 128u;
constexpr int kDwPitch = 260; // floats per row of the sums on their way out: no bank conflicts
static_assert(128 * kDwPitch * 4 <= kDwStages * kDwStageBytes, "the sums fit in the stages");
constexpr size_t kSmemDw = kDwStages * kDwStageBytes + 1024 + 256;

__global__ void __launch_bounds__(kDwThreads, 1)
    train_dw_kernel(const __grid_constant__ CUtensorMap mact, float *__restrict__ G, int64_t n_blocks,
                    int64_t blocks_per_split, int *err)
{
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    uint64_t *full = (uint64_t *)(smem + kDwStages * kDwStageBytes);
    uint64_t *empty = full + kDwStages;
    uint64_t *filled = empty + kDwStages; // [2]: a chunk's MMAs into an accumulator are complete
    uint64_t *drained = filled + 2;       // [2]: the accumulator has been read
    uint64_t *done = drained + 2;
    uint32_t *tmem_slot = (uint32_t *)(done + 1);
    volatile int *abort = (volatile int *)(tmem_slot + 1);

    const int m0 = blockIdx.y * 128, L = blockIdx.z; // L = 0..2: W2..W4
    const int64_t lo = blockIdx.x * blocks_per_split;
    const int nkb = (int)(min(n_blocks, lo + blocks_per_split) - lo);
    const int n_chunks = (nkb + kDwChunk - 1) / kDwChunk;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

    if (threadIdx.x == 0) {
        for (int s = 0; s < kDwStages; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(&filled[b], 1);
            mbar_init(&drained[b], kDwSumWarps);
        }
        mbar_init(done, 1);
        *abort = 0;
        mbar_fence_init();
    }
    if (warp == 0) {
        tmem_alloc(tmem_slot, 512);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;

    if (warp == kDwSumWarps) {
        if (lane == 0) {
            const uint32_t idesc = idesc_bf16_f32(128, 256);
            auto load = [&](int kb) {
                uint8_t *dst = smem + (kb % kDwStages) * kDwStageBytes;
                uint64_t *bar = &full[kb % kDwStages];
                const int k = (int)(lo + kb) * 64;
                mbar_expect_tx(bar, kDwStageBytes);
                tma_load_2d(dst, &mact, k, (3 + L) * 256 + m0, bar);          // dZ_{L+2}
                tma_load_2d(dst + 16384, &mact, k, L * 256, bar);             // H_{L+1}
                tma_load_2d(dst + 32768, &mact, k, L * 256 + 128, bar);
            };
            int issued = 0;
            for (; issued < nkb && issued < kDwStages; ++issued)
                load(issued);
            bool ok = true;
            for (int kb = 0; kb < nkb && ok; ++kb) {
                const int s = kb % kDwStages, c = kb / kDwChunk, b = c & 1;
                const bool first = kb % kDwChunk == 0, last = (kb + 1) % kDwChunk == 0 || kb + 1 == nkb;
                // the chunk before last, in the same accumulator, has been read
                if (first && c >= 2 && !wait_abort(&drained[b], ((c >> 1) - 1) & 1, abort, err, 43)) ok = false;
                if (!ok || !wait_abort(&full[s], (kb / kDwStages) & 1, abort, err, 41)) {
                    ok = false;
                    break;
                }
                tc_fence_after();
                const uint32_t a0 = smem_u32(smem + s * kDwStageBytes), b0 = a0 + 16384;
#pragma unroll
                for (int k = 0; k < 4; ++k)
                    mma_bf16(tmem + b * 256, desc_sw128(a0 + k * 32), desc_sw128(b0 + k * 32), idesc, (!first || k) ? 1u : 0u);
                mma_commit(&empty[s]);
                if (last) mma_commit(&filled[b]);
                // refill the stage consumed one iteration ago (its MMAs have had time to finish)
                if (kb >= 1 && kb - 1 + kDwStages < nkb) {
                    if (!wait_abort(&empty[(kb - 1) % kDwStages], ((kb - 1) / kDwStages) & 1, abort, err, 44)) {
                        ok = false;
                        break;
                    }
                    load(kb - 1 + kDwStages);
                    ++issued;
                }
            }
            // all MMAs complete, and the copies already in flight landed, before the CTA's tensor
            // and shared memory are released
            mma_commit(done);
            mbar_wait(done, 0);
            if (!ok)
                for (int j = issued > kDwStages ? issued - kDwStages : 0; j < issued; ++j)
                    mbar_wait(&full[j % kDwStages], (j / kDwStages) & 1);
        }
    } else {
        // rows 32 (warp % 4) + lane of the accumulator (the tensor-memory lanes a warp may read),
        // columns 128 (warp / 4) .. + 127
        const uint32_t ta = tmem + ((uint32_t)(warp & 3) * 32u << 16) + (uint32_t)(warp >> 2) * 128u;
        float sum[128];
#pragma unroll
        for (int i = 0; i < 128; ++i)
            sum[i] = 0.f;
        bool ok = true;
#pragma unroll 1
        for (int c = 0; c < n_chunks; ++c) {
            const int b = c & 1;
            ok = __all_sync(0xffffffffu, wait_abort(&filled[b], (c >> 1) & 1, abort, err, 42)) != 0;
            if (!ok) break;
            tc_fence_after();
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                float v[32];
                tmem_ld32(ta + (uint32_t)(b * 256 + q * 32), v);
#pragma unroll
                for (int i = 0; i < 32; ++i)
                    sum[q * 32 + i] += v[i];
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&drained[b]);
        }
        // the sums leave by rows of 1024 bytes, through the stages that are free now (every load
        // landed and was consumed before the last chunk's signal)
        float *const rows = (float *)smem;
        if (ok) {
            float *dst = rows + ((warp & 3) * 32 + lane) * kDwPitch + (warp >> 2) * 128;
#pragma unroll
            for (int j = 0; j < 32; ++j)
                reinterpret_cast<float4 *>(dst)[j] = make_float4(sum[4 * j], sum[4 * j + 1], sum[4 * j + 2], sum[4 * j + 3]);
        }
        asm volatile("bar.sync 1, %0;" ::"n"(32 * kDwSumWarps) : "memory");
        if (ok && !*abort) {
            float *dst = G + siren_oW(L + 2) + (int64_t)m0 * 256;
#pragma unroll 4
            for (int r = warp; r < 128; r += kDwSumWarps)
#pragma unroll
                for (int h = 0; h < 2; ++h)
                    atomicAdd(reinterpret_cast<float4 *>(dst + r * 256 + h * 128) + lane,
                              reinterpret_cast<const float4 *>(rows + r * kDwPitch + h * 128)[lane]);
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) {
        tc_fence_after();
        tmem_dealloc(tmem, 512);
    }
}

int sm_count()
{
    int dev = 0, n = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
    return n > 0 ? n : 1;
}

} // namespace

cudaError_t train_act_map(CUtensorMap *m, const void *act, int64_t cap)
{
    return make_map_bf16(m, act, (uint64_t)cap, 6 * 256, 128);
}

cudaError_t train_fwd_bwd(const SirenNet &net, const CUtensorMap &act, const float *x, const float *t, int64_t n,
                          float *G, double *loss, cudaStream_t s)
{
    if (n <= 0) return cudaSuccess;
    if (n % kRows != 0 || !net.err || ((uintptr_t)G & 15u) != 0) return cudaErrorInvalidValue;
    const auto fn = n <= kLibrarySines ? siren_train_kernel<true> : siren_train_kernel<false>;
    cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemTrain);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(train_dw_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemDw);
    if (e != cudaSuccess) return e;
    const int sms = sm_count();
    TrainParams p;
    p.P = net.P;
    p.W5p = (const __nv_bfloat16 *)net.W5p;
    p.x = x;
    p.t = t;
    p.n = n;
    p.omega0 = net.omega0;
    p.gscale = (float)(2.0 / (double)(n * 8));
    p.G = G;
    p.loss = loss;
    p.err = net.err;
    const int64_t tiles = n / kRows;
    fn<<<(int)(tiles < sms ? tiles : sms), kThreads, kSmemTrain, s>>>(net.map_wh, net.map_w5, act, p);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    // 6 CTAs (3 layers x 2 halves) per split of the batch: as many splits as fill the SMs once
    int64_t splits = sms / 6 > 0 ? sms / 6 : 1;
    if (splits > tiles) splits = tiles;
    const int64_t per = (tiles + splits - 1) / splits;
    splits = (tiles + per - 1) / per;
    train_dw_kernel<<<dim3((unsigned)splits, 2, 3), kDwThreads, kSmemDw, s>>>(act, G, tiles, per, net.err);
    return cudaGetLastError();
}

} // namespace gcs
