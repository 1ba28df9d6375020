// gc_siren_eval.cu -- fused evaluation of the SIREN neural field and its Jacobian on the
// tensor cores (tcgen05, TMA, tensor memory).
//
// Forward-mode differentiation carries three tangent rows beside every value row: for a
// point x the rows are h_k and t_{k,j} = dh_k/dx_j (j = 0..2), with
//   layer 1:  z = w0 (W1 x + b1),   h1 = sin z,   t1_j = w0 cos(z) W1[:, j]
//   layer k:  z = W_k h_{k-1} + b_k, h_k = sin z, t_{k,j} = cos(z) * (W_k t_{k-1,j})
//   output:   y = W5 h4 + b5,       J[:, j] = W5 t_{4,j}.
// A tile is 64 points = 256 rows (row 4p + q: q = 0 value, q = 1..3 tangents), or 16 points =
// 64 rows where that leaves every SM at most one tile (kSmallTiles). Hidden
// layers run as D = W_k . H^T on the tensor cores (two halves of M = 128 output features,
// N = 256 rows, K = 256), so that each accumulator lane holds one feature and the four rows
// of a point sit in adjacent columns: the epilogue thread of a feature computes sin and cos
// of the value row once and scales its own three tangent columns, with no data exchange.
// Activations go back to shared memory in the MN-major 128-byte-swizzled layout that the
// next layer reads as its B operand. The output layer runs as rows x W5^T (M = 128 rows,
// N = 16 with W5 zero-padded, loaded once per launch). The hidden layers' weights stream
// through a 4-stage TMA ring (16 KB chunks of 64 input features x 128 outputs; 4 stages
// measured faster than 5 or 6, 2 slower); the first layer runs on the CUDA cores.
//
// Pipeline of one layer, in MMA order: half 0 over input features 0-127, half 1 over 0-127,
// half 0 over 128-255, half 1 over 128-255. The epilogue of half 0 (features 0-127) starts
// when half 0 is complete, and with it every MMA of the layer over inputs 0-127, so it may
// overwrite them at once; it overlaps the MMAs of half 1 over 128-255. The epilogue of half
// 1 says when it has read its whole accumulator (h1_drained, halfway through): the next
// layer's MMAs over inputs 0-127 (the features half 0 has just written), half 0's during it
// and half 1's after that signal, run while it computes; those over 128-255 follow it.
// The output layer also runs in two K halves (input features 0-127 during the last
// epilogue of half 1, then 128-255) into columns 0-31 of the drained half-0 accumulator,
// and overlaps the next tile's first layer: its half 0 is written once the output MMAs over
// features 0-127 are done, and the output accumulator is read before the next tile's MMAs
// may start; the previous tile's outputs are stored while those MMAs run.
//
// Warp roles (576 threads): warps 0-15 compute; all of them work on one output half at a
// time, warp w on features 32 (w % 4) + lane of the half (warp w may only touch
// tensor-memory lanes 32 (w % 4) .. + 31) and rows 64 (w / 4) .. + 63. One lane of warp 16 issues the MMAs
// (warp 16 also owns the tensor-memory allocation), warp 17 lane 0 issues the TMA loads.
// Every wait is bounded: a wait that runs out sets the kernel's error word and an abort flag
// that makes all roles leave their loops; the CTA then waits for its own copies and MMAs
// and frees its tensor memory.
#include <cstdio>

#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include "gc_push.cuh"
#include "gc_siren.h"
#include "gc_tc.cuh"

namespace gcs {

using namespace tc;

namespace {

constexpr int kStagesW = 4;                     // weight ring depth
constexpr uint32_t kChunkBytes = 128u * 128u;   // 128 output rows x 64 bf16
constexpr uint32_t kW5Bytes = 4u * 16u * 128u;  // W5 padded: 4 boxes of 16 rows x 64 bf16
constexpr int kChunksPerTile = 3 * 8;
constexpr int kComputeWarps = 16;               // arrivals on each h_ready barrier
constexpr int kThreads = 576;
constexpr int kMmaWarp = 16, kTmaWarp = 17;
constexpr int kPushTiles = 2;   // tiles of 16 particles per SM up to which they are pushed in one launch
constexpr int kSmallTiles = 1;  // tiles of 16 points per SM up to which they are taken instead of 64
constexpr uint32_t kPtsBytes = 16u * 16u * 16u;  // per compute warp: its 16 points as float4

// A tile of PTS points (64, or 16 for few points): 4 PTS rows, a K-group of 8 features as
// blocks of 8 features x 64 rows of 1024 B
template <int PTS>
struct Tile {
    static constexpr int kRows = 4 * PTS;
    static constexpr uint32_t kGroupBytes = kRows / 64 * 1024;
    static constexpr uint32_t kHBytes = 32 * kGroupBytes;
    static constexpr int kOutTiles = kRows > 128 ? kRows / 128 : 1; // M-tiles of the output layer
    static constexpr int kWarpPts = PTS / 4, kWarpRows = kRows / 4;
    static constexpr int kCols = kWarpRows < 32 ? kWarpRows : 32; // columns per tensor-memory load
    static constexpr uint32_t kTmemCols = 2 * kRows;
    static constexpr size_t kSmem = kHBytes + kStagesW * kChunkBytes + kW5Bytes + kPtsBytes + 1024 + 256;
};

struct EvalParams {
    const float *P;  // master parameters
    SirenIn in;
    SirenOut out;
    float omega0;
    int *err;        // error word (device), set when a wait runs out
};

// 8 consecutive rows (mn0 .. mn0 + 7, mn0 % 8 == 0) of one feature into the MN-major
// activation buffer; hrow points at the feature's 128-byte row of its K-group's first atom
__device__ __forceinline__ void store_rows8(uint8_t *hrow, uint32_t rsw, uint32_t mn0, const float (&o)[8])
{
    uint4 pk;
    pk.x = pack_bf16(o[0], o[1]);
    pk.y = pack_bf16(o[2], o[3]);
    pk.z = pack_bf16(o[4], o[5]);
    pk.w = pack_bf16(o[6], o[7]);
    const uint32_t ch = ((mn0 & 63u) >> 3) ^ rsw;
    *reinterpret_cast<uint4 *>(hrow + (mn0 >> 6) * 1024u + ch * 16u) = pk;
}

// Physical field at R = (X0, X1, X2) from row q (0 value, 1..3 tangents) v of the output and the
// point's values yv: B = B_s y_B (AU/r)^2, E = E_s y_E (AU/r); gradients by the product rule
// with d/dR = (x_scale / pos_scale) d/dx.
__device__ __forceinline__ void field_row(const EvalParams &p, int q, const float (&yv)[6], const float (&v)[16], float X0,
                                          float X1, float X2, float *dst)
{
    const double au = 1.495978707e11;
    const float ps = p.in.pos_scale;
    const float r2 = X0 * X0 + X1 * X1 + X2 * X2;
    const float ir = rsqrtf(r2);
    const float a = (float)au * ir;                   // AU / r
    const float bs = (float)p.out.B_scale * a * a;    // B per unit y_B
    const float es = (float)p.out.E_scale * a;        // E per unit y_E
    if (q == 0) {
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            dst[c] = bs * yv[c];
            dst[3 + c] = es * yv[3 + c];
        }
    } else {
        const int d = q - 1;
        const float Xd = d == 0 ? X0 : (d == 1 ? X1 : X2);
        const float irm = p.in.x_scale / ps;  // d/dR = (x_scale / pos_scale) d/dx
        const float ur = Xd * ir * ir;  // R_d / r^2
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            dst[6 + 3 * d + c] = bs * (v[c] * irm - 2.0f * yv[c] * ur);
            dst[15 + 3 * d + c] = es * (v[3 + c] * irm - yv[3 + c] * ur);
        }
        // the push's layout also takes grad(Phi): Phi = E_scale AU y_Phi
        if (p.out.field_stride >= 40)
            dst[34 + d] = (float)(p.out.E_scale * au) * v[7] * irm;
    }
}

// values of the point that this lane's row belongs to (lanes 4 p .. 4 p + 3 hold its rows)
__device__ __forceinline__ void point_values(const float (&b5)[8], const float (&v)[16], int lane, float (&yv)[6])
{
#pragma unroll
    for (int o = 0; o < 6; ++o)
        yv[o] = __shfl_sync(0xffffffffu, v[o] + b5[o], lane & ~3);
}

// Output rows of one tile from the output accumulator v (16 columns of this thread's row
// pr): raw outputs y and J, or the physical field for the push.
__device__ __forceinline__ void store_out(const EvalParams &p, const float (&b5)[8], const float (&v)[16],
                                          int64_t base, int pr, int lane, int64_t n_pts)
{
    const int q = pr & 3;
    const int64_t P = base + (pr >> 2);
    if (p.out.field == nullptr) {
        if (P < n_pts) {
            if (q == 0) {
#pragma unroll
                for (int o = 0; o < 8; ++o)
                    p.out.y[P * 8 + o] = v[o] + b5[o];
            } else if (p.out.J) {
#pragma unroll
                for (int o = 0; o < 8; ++o)
                    p.out.J[(P * 8 + o) * 3 + (q - 1)] = v[o];
            }
        }
    } else {
        float yv[6];
        point_values(b5, v, lane, yv);
        if (P < n_pts) {
            const float ps = p.in.pos_scale;
            field_row(p, q, yv, v, __ldg(p.in.p + 3 * P) * ps, __ldg(p.in.p + 3 * P + 1) * ps,
                      __ldg(p.in.p + 3 * P + 2) * ps, p.out.field + P * p.out.field_stride);
        }
    }
}

// Rows of the first layer for kPairs pairs of points pts[0 ..] into one half's features
template <int kPairs>
__device__ __forceinline__ void layer1_rows(const float4 *pts, float w0, const float (&w)[3], float b, uint8_t *hrow,
                                            uint32_t rsw, uint32_t row0)
{
#pragma unroll 2
    for (int p2 = 0; p2 < kPairs; ++p2) {
        float o[8];
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            const float4 xq = pts[2 * p2 + e];
            const float x0 = xq.x, x1 = xq.y, x2 = xq.z;
            const float z = w0 * fmaf(w[0], x0, fmaf(w[1], x1, fmaf(w[2], x2, b)));
            // the hardware sine and cosine on z directly (|z| reaches tens here, w0
            // = 30): their error, a few 1e-6 at most there, stays three orders below
            // the BF16 rounding of the activations; an explicit reduction by 2 pi
            // first cost 2 % of the kernel for no gain against the exact network
            const float sn = __sinf(z), cs = __cosf(z);
            const float wc = w0 * cs;
            o[4 * e] = sn;
            o[4 * e + 1] = wc * w[0];
            o[4 * e + 2] = wc * w[1];
            o[4 * e + 3] = wc * w[2];
        }
        store_rows8(hrow, rsw, row0 + 8 * p2, o);
    }
}

// Rows row0 .. row0 + N - 1 of a hidden layer's output from the accumulator columns v
template <int N>
__device__ __forceinline__ void hidden_rows(const float (&v)[N], float b, uint8_t *hrow, uint32_t rsw, uint32_t row0)
{
    float o[N / 8][8];
#pragma unroll
    for (int pp = 0; pp < N / 8; ++pp)
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            // |z| stays small in the hidden layers: the hardware sine
            // and cosine without a range reduction
            const int q0 = 8 * pp + 4 * e;
            const float z = v[q0] + b;
            const float sn = __sinf(z), cs = __cosf(z);
            o[pp][4 * e] = sn;
            o[pp][4 * e + 1] = cs * v[q0 + 1];
            o[pp][4 * e + 2] = cs * v[q0 + 2];
            o[pp][4 * e + 3] = cs * v[q0 + 3];
        }
#pragma unroll
    for (int pp = 0; pp < N / 8; ++pp)
        store_rows8(hrow, rsw, row0 + 8 * pp, o[pp]);
}

// What the roles of a CTA share: operand buffers and barriers in shared memory.
struct Roles {
    uint8_t *sH, *sW, *sW5;  // activations, weight ring, W5 (resident for the whole launch)
    uint64_t *full, *empty;  // [stages]
    uint64_t *h_ready;       // [2]: activations of a half written, its accumulator drained
    uint64_t *acc;           // [2]: accumulator of a half complete
    uint64_t *h1_drained;    // the half-1 epilogue has read its accumulator
    uint64_t *acc_out;       // output layer complete
    uint64_t *out_a;         // output-layer MMAs over input features 0-127 complete
    uint64_t *fin;
    uint64_t *w5full;        // W5 landed
    volatile int *abort;     // 1: a wait ran out; 2: the CTA's work is done (roles without a count)
};

// Weight loads of `rounds` evaluations of a tile (one thread); ends early on the abort flag.
// kForever rounds end when the flag is up after a wait: who raises it completes the barriers that
// the roles wait on (pts_ready; the compute warps h_ready[0]; the MMA warp the empty stages).
constexpr int64_t kForever = INT64_MAX;

template <int STAGES>
__device__ __forceinline__ void load_role(const Roles &R, const CUtensorMap &mwh, const CUtensorMap &mw5, int64_t rounds,
                                          int *err)
{
    if ((threadIdx.x & 31) != 0) return;
    uint32_t st = 0, par = 1, filled = 0;
    bool ok = true;
    mbar_expect_tx(R.w5full, kW5Bytes);
    for (int kb = 0; kb < 4; ++kb)
        tma_load_2d(R.sW5 + kb * 2048, &mw5, kb * 64, 0, R.w5full);
    for (int64_t r = 0; r < rounds && ok; ++r) {
#pragma unroll 1
        for (int c = 0; c < kChunksPerTile; ++c) {
            if (!wait_abort(&R.empty[st], par, R.abort, err, 11) || (rounds == kForever && *R.abort)) {
                ok = false;
                break;
            }
            // chunk (layer c / 8, output half and input block in the MMA order)
            const int q = c & 7, h = (q >> 1) & 1, kb = (q & 1) | ((q >> 2) << 1);
            mbar_expect_tx(&R.full[st], kChunkBytes);
            tma_load_2d(R.sW + st * kChunkBytes, &mwh, kb * 64, (c >> 3) * 256 + h * 128, &R.full[st]);
            filled |= 1u << st;
            if (++st == STAGES) {
                st = 0;
                par ^= 1u;
            }
        }
    }
    // the copies still in flight land before the CTA's shared memory is released: the
    // last copy of a stage behind st is of the running phase, of one from st on of the
    // phase before
    for (int j = 0; j < STAGES; ++j)
        if (filled >> j & 1)
            mbar_wait(&R.full[j], (uint32_t)j < st ? par ^ 1u : par);
    mbar_wait(R.w5full, 0);
}

// MMAs of `rounds` evaluations (the whole warp); ends early on the abort flag.
template <class Tl, int STAGES>
__device__ __forceinline__ void mma_role(const Roles &R, uint32_t tmem, int64_t rounds, int *err)
{
    constexpr uint32_t kGroup = Tl::kGroupBytes;
    // The whole warp runs the loop and one elected lane issues; descriptors are a constant
    // high word and a running low word. With descriptors built from addresses for every MMA
    // and the stage found by a division, beside four compute warps on the same scheduler an
    // MMA took 170 cycles to issue against the 128 the tensor cores need for it.
    constexpr uint32_t id_hid = idesc_bf16_f32(128, Tl::kRows, 0, 1);
    constexpr uint32_t id_out = idesc_bf16_f32(128, 16, 1, 0);
    const bool leader = elect_one();
    const uint32_t tm = __shfl_sync(0xffffffffu, tmem, 0);
    const uint32_t h_lo = desc_lo(smem_u32(R.sH), 1024), w_lo = desc_lo(smem_u32(R.sW), 16);
    uint32_t st = 0, par = 0, nh = 0, nd = 0; // ring stage and its phase, operands, drains
    bool ok = true;
    auto wait = [&](uint64_t *bar, uint32_t phase, int code) {
        const bool done = __all_sync(0xffffffffu, wait_abort(bar, phase & 1u, R.abort, err, code)) != 0;
        tc_fence_after();
        return done && !(rounds == kForever && *R.abort);
    };
    // W5, loaded once per launch
    if (rounds > 0) ok = wait(R.w5full, 0, 17);
    for (int64_t r = 0; r < rounds && ok; ++r) {
#pragma unroll 1
        for (int L = 0; L < 3 && ok; ++L) {
            // order: half 0 over inputs 0-127, half 1 over inputs 0-127 (as soon as the
            // previous half-1 epilogue has read its accumulator), half 0 over 128-255
            // (once that epilogue has written them), half 1 over 128-255
#pragma unroll 1
            for (int q = 0; q < 8; ++q) {
                const int h = (q >> 1) & 1, kb = (q & 1) | ((q >> 2) << 1);
                // inputs 0-127 written and accumulator half 0 drained
                if (q == 0 && !wait(&R.h_ready[0], nh, 12)) { ok = false; break; }
                if (q == 2 && (L > 0 || r > 0)) {
                    // accumulator half 1 read by the previous half-1 epilogue
                    if (!wait(R.h1_drained, nd, 19)) { ok = false; break; }
                    ++nd;
                }
                // inputs 128-255 written
                if (q == 4 && !wait(&R.h_ready[1], nh, 13)) { ok = false; break; }
                if (!wait(&R.full[st], par, 14)) { ok = false; break; }
                if (leader) {
                    const uint32_t a_lo = w_lo + st * (kChunkBytes / 16), b_lo = h_lo + kb * (8 * kGroup / 16);
#pragma unroll
                    for (int ks = 0; ks < 4; ++ks)
                        mma_bf16(tm + h * Tl::kRows, desc_of(desc_hi(1024), a_lo + ks * (32 / 16)),
                                 desc_of(desc_hi(kGroup), b_lo + ks * (2 * kGroup / 16)), id_hid,
                                 (uint32_t)(kb | ks));
                    mma_commit(&R.empty[st]);
                    // half 0 complete, and with it every MMA of this layer over inputs 0-127
                    if (q == 5) mma_commit(&R.acc[0]);
                    if (q == 7) mma_commit(&R.acc[1]);
                }
                __syncwarp();
                if (++st == STAGES) {
                    st = 0;
                    par ^= 1u;
                }
            }
            ++nh;
        }
        // output layer: rows x W5^T, M-tile 0 into columns 0-15 and M-tile 1 into 16-31
        // (both in the drained half-0 accumulator; of a 64-row tile's one M-tile the upper
        // 64 rows read on into the next features, or the ring, and are not used), in two K halves: input features
        // 0-127 as soon as their epilogue is done, 128-255 after the last one
        for (int kh = 0; kh < 2 && ok; ++kh) {
            if (!wait(&R.h_ready[kh], nh, 15 + kh)) { ok = false; break; }
            if (leader) {
                const uint32_t w5_lo = desc_lo(smem_u32(R.sW5), 16);
#pragma unroll
                for (int mt = 0; mt < Tl::kOutTiles; ++mt)
#pragma unroll
                    for (int k8 = 0; k8 < 8; ++k8) {
                        const int k16 = kh * 8 + k8;
                        mma_bf16(tm + mt * 16, desc_of(desc_hi(kGroup), h_lo + (mt * 2048 + k16 * 2 * kGroup) / 16),
                                 desc_of(desc_hi(1024), w5_lo + ((k16 >> 2) * 2048 + (k16 & 3) * 32) / 16), id_out,
                                 k16 ? 1u : 0u);
                    }
                mma_commit(kh ? R.acc_out : R.out_a);
            }
            __syncwarp();
        }
        ++nh;
    }
    // all MMAs of this CTA complete before its tensor memory is released
    if (leader) {
        mma_commit(R.fin);
        mbar_wait(R.fin, 0);
        if (rounds == kForever)
            for (int j = 0; j < STAGES; ++j)
                mbar_arrive(&R.empty[j]);
    }
    __syncwarp();
}

template <int PTS>
__global__ void __launch_bounds__(kThreads, 1)
    siren_eval_kernel(const __grid_constant__ CUtensorMap mwh, const __grid_constant__ CUtensorMap mw5,
                      const __grid_constant__ EvalParams p)
{
    using Tl = Tile<PTS>;
    constexpr uint32_t kGroup = Tl::kGroupBytes;
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    uint8_t *sH = smem;
    uint8_t *sW = smem + Tl::kHBytes;
    uint8_t *sW5 = sW + kStagesW * kChunkBytes;  // W5, resident for the whole launch
    float4 *sPts = (float4 *)(sW5 + kW5Bytes);  // [16 compute warps][16 points]
    uint64_t *full = (uint64_t *)(sW5 + kW5Bytes + kPtsBytes);
    uint64_t *empty = full + kStagesW;
    uint64_t *h_ready = empty + kStagesW; // [2]: activations of a half written, its accumulator drained
    uint64_t *acc = h_ready + 2;          // [2]: accumulator of a half complete
    uint64_t *h1_drained = acc + 2;       // the half-1 epilogue has read its accumulator
    uint64_t *acc_out = h1_drained + 1;   // output layer complete
    uint64_t *out_a = acc_out + 1;        // output-layer MMAs over input features 0-127 complete
    uint64_t *fin = out_a + 1;
    uint64_t *w5full = fin + 1;           // W5 landed
    uint32_t *tmem_slot = (uint32_t *)(w5full + 1);
    volatile int *abort = (volatile int *)(tmem_slot + 1);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    int64_t n_pts = p.in.n;
    if (p.in.n_dev) {
        const int64_t nd = *p.in.n_dev;
        n_pts = nd < n_pts ? (nd > 0 ? nd : 0) : n_pts;
    }
    const int64_t n_tiles = (n_pts + PTS - 1) / PTS;
    const int64_t n_rounds = blockIdx.x < n_tiles ? (n_tiles - blockIdx.x + gridDim.x - 1) / gridDim.x : 0;
    const Roles R{sH, sW, sW5, full, empty, h_ready, acc, h1_drained, acc_out, out_a, fin, w5full, abort};

    if (threadIdx.x == 0) {
        for (int s = 0; s < kStagesW; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        mbar_init(&h_ready[0], kComputeWarps);
        mbar_init(&h_ready[1], kComputeWarps);
        mbar_init(&acc[0], 1);
        mbar_init(&acc[1], 1);
        mbar_init(h1_drained, kComputeWarps);
        mbar_init(acc_out, 1);
        mbar_init(out_a, 1);
        mbar_init(fin, 1);
        mbar_init(w5full, 1);
        *abort = 0;
        mbar_fence_init();
    }
    if (warp == kMmaWarp) {
        tmem_alloc(tmem_slot, Tl::kTmemCols);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;

    if (warp == kTmaWarp) {
        load_role<kStagesW>(R, mwh, mw5, n_rounds, p.err);
    } else if (warp == kMmaWarp) {
        mma_role<Tl, kStagesW>(R, tmem, n_rounds, p.err);
    } else {
        // ------------------------------------------------------------ compute warps
        // warp w: tensor-memory lane quarter lq = w % 4 (features 32 lq .. of each half) and
        // row group rg = w / 4 (rows 64 rg .. 64 rg + 63 = points 16 rg .. 16 rg + 15); all
        // 16 warps work on one output half at a time
        const int lq = warp & 3, rg = warp >> 2;
        const float w0 = p.omega0;
        float w1[2][3], b1[2], bl[3][2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int f = h * 128 + lq * 32 + lane;
#pragma unroll
            for (int j = 0; j < 3; ++j)
                w1[h][j] = p.P[siren_oW(1) + 3 * f + j];
            b1[h] = p.P[siren_oB(1) + f];
#pragma unroll
            for (int L = 0; L < 3; ++L)
                bl[L][h] = p.P[siren_oB(L + 2) + f];
        }
        float b5[8];
#pragma unroll
        for (int o = 0; o < 8; ++o)
            b5[o] = p.P[siren_oB(5) + o];
        const uint32_t lane_base = tmem + ((uint32_t)(lq * 32) << 16);
        // the feature's 128-byte row in its K-group's first atom, for each half
        uint8_t *hrow0 = sH + ((lq * 32 + lane) >> 3) * kGroup + (lane & 7) * 128;
        uint8_t *hrow1 = hrow0 + 16 * kGroup;
        const uint32_t rsw = (uint32_t)(lane & 7);
        uint32_t na0 = 0, na1 = 0, no = 0, noa = 0;
        bool ok = true, first = true;
        int64_t base_prev = 0;
        // this warp's 16 points: lane i < 16 holds point 16 rg + i and puts it in the warp's
        // shared-memory slots for the first layer, where every lane reads it by broadcast; the
        // next tile's are fetched while the current one runs
        float px = 0.f, py = 0.f, pz = 0.f;
        const int pt_off = rg * Tl::kWarpPts + (lane & (Tl::kWarpPts - 1));
        // this warp's part of the output accumulator (its M-tile rg)
        const bool outs = rg < Tl::kOutTiles && lq * 32 < Tl::kRows;
        {
            const int64_t P = (int64_t)blockIdx.x * PTS + pt_off;
            if (P < n_pts) {
                px = __ldg(p.in.p + 3 * P) * p.in.x_scale;
                py = __ldg(p.in.p + 3 * P + 1) * p.in.x_scale;
                pz = __ldg(p.in.p + 3 * P + 2) * p.in.x_scale;
            }
        }
        float4 *wpts = sPts + warp * 16;
        for (int64_t t = blockIdx.x; t < n_tiles && ok; t += gridDim.x) {
            const int64_t base = t * PTS;
            __syncwarp();  // every lane done with the previous tile's points
            if (lane < Tl::kWarpPts) wpts[lane] = make_float4(px, py, pz, 0.f);
            __syncwarp();
            // Layer 1 on the CUDA cores, half 0 then half 1. The previous tile's output layer
            // still runs meanwhile: half 0 overwrites input features 0-127 once the output
            // MMAs over them are done (out_a); before half 0 is announced, the output
            // accumulator is read (the next MMAs overwrite it); half 1 follows the rest of the
            // output layer (acc_out), then the previous tile's outputs are stored.
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                uint8_t *hrow = h ? hrow1 : hrow0;
                if (h == 0 && !first) {
                    if (!wait_abort(out_a, noa & 1u, abort, p.err, 21)) {
                        ok = false;
                        break;
                    }
                    ++noa;
                }
                layer1_rows<Tl::kWarpPts / 2>(wpts, w0, w1[h], b1[h], hrow, rsw, (uint32_t)(rg * Tl::kWarpRows));
                fence_proxy_async_smem();
                float v[16];
                if (h == 0 && !first) {
                    if (!wait_abort(acc_out, no & 1u, abort, p.err, 20)) {
                        ok = false;
                        break;
                    }
                    ++no;
                    tc_fence_after();
                    if (outs) tmem_ld16(lane_base + rg * 16, v);
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&h_ready[h]);
                if (h == 0 && !first && outs)
                    store_out(p, b5, v, base_prev, rg * 128 + lq * 32 + lane, lane, n_pts);
            }
            if (!ok) break;
            {
                const int64_t P = (t + gridDim.x) * PTS + pt_off;
                px = py = pz = 0.f;
                if (t + gridDim.x < n_tiles && P < n_pts) {
                    px = __ldg(p.in.p + 3 * P) * p.in.x_scale;
                    py = __ldg(p.in.p + 3 * P + 1) * p.in.x_scale;
                    pz = __ldg(p.in.p + 3 * P + 2) * p.in.x_scale;
                }
            }
            // hidden layers 2-4: epilogues of D = W_k H^T, half 0 then half 1
            for (int L = 0; L < 3 && ok; ++L) {
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    uint32_t &na = h ? na1 : na0;
                    if (!wait_abort(&acc[h], na & 1u, abort, p.err, 18)) {
                        ok = false;
                        break;
                    }
                    ++na;
                    tc_fence_after();
                    uint8_t *hrow = h ? hrow1 : hrow0;
                    const float b = bl[L][h];
                    // (half 0: every MMA over inputs 0-127 is complete with its accumulator)
#pragma unroll 1
                    for (int c = 0; c < Tl::kWarpRows / Tl::kCols; ++c) {
                        float v[Tl::kCols];
                        tmem_ld(lane_base + h * Tl::kRows + rg * Tl::kWarpRows + c * Tl::kCols, v);
                        if (h == 1 && c == Tl::kWarpRows / Tl::kCols - 1) {
                            // the half-1 accumulator is read: the next layer's half-1 MMAs
                            // over inputs 0-127 may run during the rest of this epilogue
                            tc_fence_before();
                            __syncwarp();
                            if (lane == 0) mbar_arrive(h1_drained);
                        }
                        hidden_rows(v, b, hrow, rsw, (uint32_t)(rg * Tl::kWarpRows + c * Tl::kCols));
                    }
                    fence_proxy_async_smem();
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&h_ready[h]);
                }
            }
            if (!ok) break;
            base_prev = base;
            first = false;
        }
        // the last tile's output layer
        if (ok && !first && wait_abort(acc_out, no & 1u, abort, p.err, 20)) {
            tc_fence_after();
            if (outs) {
                float v[16];
                tmem_ld16(lane_base + rg * 16, v);
                store_out(p, b5, v, base_prev, rg * 128 + lq * 32 + lane, lane, n_pts);
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == kMmaWarp) {
        tc_fence_after();
        tmem_dealloc(tmem, Tl::kTmemCols);
    }
}

// ----------------------------------------------------------------------------------------
// The neural push of a small population in one launch: a CTA owns 16 particles at a time and
// takes them through all the launch's steps, one warp pushing them (a lane per particle, state in
// registers) and the other roles evaluating the network at their requests as above, with
// requests and samples in shared memory. Each particle walks its phases at its own pace (see
// the split-step push), so the tile runs 2 n_steps evaluations plus two per event of its
// unluckiest particle. What bounds it is the latency of one evaluation and one push phase.
constexpr int kPushPts = 16, kPushStages = 8, kPushWarp = 18, kPushThreads = 608;
using PushTile = Tile<kPushPts>;
constexpr uint32_t kSampleBytes = kPushPts * gcp::kSampleStride * 4;
constexpr size_t kPushSmem =
    PushTile::kHBytes + kPushStages * kChunkBytes + kW5Bytes + kPushPts * 16 + kSampleBytes + 1024 + 512;

__global__ void __launch_bounds__(kPushThreads, 1)
    siren_push_kernel(const __grid_constant__ CUtensorMap mwh, const __grid_constant__ CUtensorMap mw5,
                      const __grid_constant__ EvalParams p, const __grid_constant__ gcp::Phys<float> ph,
                      const __grid_constant__ gcp::PushParams P, int ideal)
{
    using Tl = PushTile;
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    uint8_t *sH = smem, *sW = smem + Tl::kHBytes, *sW5 = sW + kPushStages * kChunkBytes;
    float4 *sPts = (float4 *)(sW5 + kW5Bytes);            // [16] requests (m), then scaled by x_scale
    float *sS = (float *)(sPts + kPushPts);               // [16][kSampleStride] samples
    uint64_t *full = (uint64_t *)((uint8_t *)sS + kSampleBytes);
    uint64_t *empty = full + kPushStages;
    uint64_t *h_ready = empty + kPushStages, *acc = h_ready + 2, *h1_drained = acc + 2, *acc_out = h1_drained + 1,
             *out_a = acc_out + 1, *fin = out_a + 1, *w5full = fin + 1;
    uint64_t *pts_ready = w5full + 1; // the tile's next requests are in sPts
    uint64_t *out_ready = pts_ready + 1; // their samples are in sS
    uint32_t *tmem_slot = (uint32_t *)(out_ready + 1);
    volatile int *abort = (volatile int *)(tmem_slot + 1);
    const Roles R{sH, sW, sW5, full, empty, h_ready, acc, h1_drained, acc_out, out_a, fin, w5full, abort};

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        for (int s = 0; s < kPushStages; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        for (int h = 0; h < 2; ++h) {
            mbar_init(&h_ready[h], kComputeWarps);
            mbar_init(&acc[h], 1);
        }
        mbar_init(h1_drained, kComputeWarps);
        mbar_init(acc_out, 1);
        mbar_init(out_a, 1);
        mbar_init(fin, 1);
        mbar_init(w5full, 1);
        mbar_init(pts_ready, 1);
        mbar_init(out_ready, 2);
        *abort = 0;
        mbar_fence_init();
    }
    if (warp == kMmaWarp) {
        tmem_alloc(tmem_slot, Tl::kTmemCols);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    auto wait = [&](uint64_t *bar, uint32_t phase, int code) {
        return __all_sync(0xffffffffu, wait_abort(bar, phase & 1u, abort, p.err, code)) != 0;
    };

    if (warp == kTmaWarp) {
        load_role<kPushStages>(R, mwh, mw5, kForever, p.err);
    } else if (warp == kMmaWarp) {
        mma_role<Tl, kPushStages>(R, tmem, kForever, p.err);
    } else if (warp == kPushWarp) {
        // ------------------------------------------------------------ push warp
        using Acc = gcp::AccOf<float>;
        const float dtT = (float)P.dt;
        const gcp::StepW<float> w1 = {dtT * 1.5f, dtT * -0.5f, dtT * (float)(2.0 / 3.0), dtT * (float)(5.0 / 12.0),
                                      dtT * (float)(-1.0 / 12.0)};
        unsigned n_coll = 0, n_reb = 0;
        uint32_t n_out = 0;
        bool ok = true;
        for (int64_t t = blockIdx.x; t * kPushPts < P.st.n && ok; t += gridDim.x) {
            const int64_t i = t * kPushPts + lane;
            const bool mine = lane < kPushPts && i < P.st.n;
            gcp::PConst c;
            gcp::PState<float> s;
            int step = P.n_steps, phase = 0;
            float px = 1.0e11f, py = 0.f, pz = 0.f, pu; // lanes without a particle: any point
            if (mine) {
                gcp::load_particle(P, i, c, s);
                gcp::phase_point(0, s, gcp::step_weights(w1, dtT, s.hprev), dtT, px, py, pz, pu);
                step = 0;
            }
            while (ok && __any_sync(0xffffffffu, step < P.n_steps)) {
                if (lane < kPushPts) sPts[lane] = make_float4(px, py, pz, 0.f);
                __syncwarp();
                if (lane == 0) mbar_arrive(pts_ready);
                ok = wait(out_ready, n_out++, 24);
                if (ok && step < P.n_steps) {
                    gcp::Sample<float> smp;
                    gcp::load_sample<true>(sS, lane, 0, smp);
                    gcp::sampled_phase(P, ph, ideal, i, s, c, smp, w1, dtT, P.kbase, step, phase, px, py, pz, n_coll, n_reb);
                }
                __syncwarp();
            }
            if (ok && mine) gcp::store_particle(P, i, s);
            __syncwarp();
        }
        gcp::flush_counters(P, n_coll, n_reb);
        // the other roles leave their waits
        __syncwarp();
        if (lane == 0) {
            if (*abort == 0) *abort = 2;
            __threadfence_block();
            mbar_arrive(pts_ready);
        }
    } else {
        // ------------------------------------------------------------ compute warps
        const int lq = warp & 3, rg = warp >> 2;
        const float w0 = p.omega0;
        float w1[2][3], b1[2], bl[3][2], b5[8];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int f = h * 128 + lq * 32 + lane;
#pragma unroll
            for (int j = 0; j < 3; ++j)
                w1[h][j] = p.P[siren_oW(1) + 3 * f + j];
            b1[h] = p.P[siren_oB(1) + f];
#pragma unroll
            for (int L = 0; L < 3; ++L)
                bl[L][h] = p.P[siren_oB(L + 2) + f];
        }
#pragma unroll
        for (int o = 0; o < 8; ++o)
            b5[o] = p.P[siren_oB(5) + o];
        const uint32_t lane_base = tmem + ((uint32_t)(lq * 32) << 16);
        uint8_t *hrow0 = sH + ((lq * 32 + lane) >> 3) * Tl::kGroupBytes + (lane & 7) * 128;
        const uint32_t rsw = (uint32_t)(lane & 7), row0 = (uint32_t)(rg * Tl::kWarpRows);
        auto announce = [&](int h) {
            fence_proxy_async_smem();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&h_ready[h]);
        };
        uint32_t na = 0;
        for (uint32_t r = 0;; ++r) {
            if (!wait(pts_ready, r, 25) || *abort) {
                if (lane == 0) mbar_arrive(&h_ready[0]);
                break;
            }
            tc_fence_after();
            float4 pts[Tl::kWarpPts];
#pragma unroll
            for (int k = 0; k < Tl::kWarpPts; ++k) {
                const float4 q = sPts[rg * Tl::kWarpPts + k];
                pts[k] = make_float4(q.x * p.in.x_scale, q.y * p.in.x_scale, q.z * p.in.x_scale, 0.f);
            }
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                layer1_rows<Tl::kWarpPts / 2>(pts, w0, w1[h], b1[h], hrow0 + h * 16 * Tl::kGroupBytes, rsw, row0);
                announce(h);
            }
            bool ok = true;
#pragma unroll
            for (int L = 0; L < 3; ++L)
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    ok = ok && wait(&acc[h], na, 18);
                    if (!ok) break;
                    na += h;
                    tc_fence_after();
                    float v[Tl::kCols];
                    tmem_ld(lane_base + h * Tl::kRows + row0, v);
                    if (h == 1) {
                        tc_fence_before();
                        __syncwarp();
                        if (lane == 0) mbar_arrive(h1_drained);
                    }
                    hidden_rows(v, bl[L][h], hrow0 + h * 16 * Tl::kGroupBytes, rsw, row0);
                    announce(h);
                }
            if (!ok) break;
            if (rg == 0 && lq < 2) {
                // rows 32 lq + lane: point 8 lq + lane / 4
                if (!wait(acc_out, r, 20)) break;
                tc_fence_after();
                float v[16], yv[6];
                tmem_ld16(lane_base, v);
                tc_fence_before();
                point_values(b5, v, lane, yv);
                const int k = lq * 8 + (lane >> 2);
                const float4 q = sPts[k];
                const float ps = p.in.pos_scale;
                field_row(p, lane & 3, yv, v, q.x * ps, q.y * ps, q.z * ps, sS + k * gcp::kSampleStride);
                __syncwarp();
                if (lane == 0) mbar_arrive(out_ready);
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == kMmaWarp) {
        tc_fence_after();
        tmem_dealloc(tmem, Tl::kTmemCols);
    }
}

} // namespace

cudaError_t siren_maps(SirenNet &net)
{
    cudaError_t e = make_map_bf16(&net.map_wh, net.Wh, 256, 3 * 256, 128);
    if (e == cudaSuccess) e = make_map_bf16(&net.map_w5, net.W5p, 256, 16, 16);
    return e;
}

namespace {

int sm_count()
{
    static int n_sm = 0;
    if (!n_sm) {
        int dev = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev);
        if (n_sm <= 0) n_sm = 1;
    }
    return n_sm;
}

template <int PTS>
cudaError_t launch_eval(const SirenNet &net, const EvalParams &p, int64_t n, cudaStream_t s)
{
    cudaError_t e = cudaFuncSetAttribute(siren_eval_kernel<PTS>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)Tile<PTS>::kSmem);
    if (e != cudaSuccess) return e;
    const int64_t tiles = (n + PTS - 1) / PTS;
    const int grid = (int)(tiles < sm_count() ? tiles : sm_count());
    siren_eval_kernel<PTS><<<grid, kThreads, Tile<PTS>::kSmem, s>>>(net.map_wh, net.map_w5, p);
    return cudaGetLastError();
}

} // namespace

cudaError_t siren_eval(const SirenNet &net, const SirenIn &in, const SirenOut &out, cudaStream_t s)
{
    if (in.n <= 0) return cudaSuccess;
    if (!net.err) return cudaErrorInvalidValue;
    EvalParams p;
    p.P = net.P;
    p.in = in;
    p.out = out;
    p.omega0 = net.omega0;
    p.err = net.err;
    // Few points: tiles of 16 spread over the SMs and pass the chain of layers sooner. A count on
    // the device may be as large as its capacity (the particles that events have held up in the
    // split-step push), so the capacity decides (200 000 particles, three events each in 8 steps:
    // 1.32 ns a point, 1.29 without events; 1.92 with tiles of 16 for every count on the device).
    if (in.n <= (int64_t)kSmallTiles * 16 * sm_count()) return launch_eval<16>(net, p, in.n, s);
    return launch_eval<64>(net, p, in.n, s);
}

bool siren_push_fits(int64_t n) { return n <= (int64_t)kPushTiles * kPushPts * sm_count(); }

cudaError_t siren_push(const SirenNet &net, const SirenIn &in, const SirenOut &out, const gcp::PhysHost &phys,
                       const gcp::PushParams &push, int ideal, cudaStream_t s)
{
    if (push.st.n <= 0) return cudaSuccess;
    if (!net.err) return cudaErrorInvalidValue;
    cudaError_t e = cudaFuncSetAttribute(siren_push_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kPushSmem);
    if (e != cudaSuccess) return e;
    EvalParams p;
    p.P = net.P;
    p.in = in;
    p.out = out;
    p.omega0 = net.omega0;
    p.err = net.err;
    const int64_t tiles = (push.st.n + kPushPts - 1) / kPushPts;
    const int grid = (int)(tiles < sm_count() ? tiles : sm_count());
    siren_push_kernel<<<grid, kPushThreads, kPushSmem, s>>>(net.map_wh, net.map_w5, p, gcp::make_phys<float>(phys), push,
                                                            ideal);
    return cudaGetLastError();
}

} // namespace gcs
