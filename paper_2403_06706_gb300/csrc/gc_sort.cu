// gc_sort.cu -- counting sort of the particle structure-of-arrays by coarse grid cell.
//
// Particles that share grid cells then share warps, so the eight corner records of a
// field gather hit the same L1/L2 lines. The sort does not change any result: every
// random draw is keyed by the particle id and every tally is an integer sum.
//   1. key: coarse cell of each particle; rank: its slot in the bin (atomic counter)
//   2. exclusive scan of the bin counts within blocks of kScanBins bins, and the blocks' sums
//   3. destination slot of each particle: block offset + offset[key] + rank
//   4. every state array moved to the destinations, one array after the other, then a pointer
//      swap
// What bounds it is memory traffic (344 bytes a particle to move). The key only groups
// particles, so it is computed in FP32 (FP64 arctangents took half of the sort). Arrays move
// one by one because a destination array up to the L2's size is then written whole there,
// while 24 arrays at once evict partly written sectors. A sort of 3 x 10^6 particles in state
// order takes 0.22 ms (1.42 before, 0.15 at the copy rate), the copy back into id order 0.4
// (1.1 to 1.6 before).
#include <algorithm>

#include "gc_device.cuh"
#include "gc_sort.h"

namespace gcp {

namespace {

struct KeyGeom {
    float r_min, inv_dr, inv_dth, inv_dph;
    int n_r, n_th, n_ph, shift;
    int nr_c, nth_c, nph_c;
};

__global__ void key_kernel(const double *__restrict__ x, const double *__restrict__ y,
                           const double *__restrict__ z, int64_t n, KeyGeom g, uint32_t *key,
                           uint32_t *rank, uint32_t *hist)
{
    const unsigned lane = threadIdx.x & 31u;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        const float X = (float)x[i], Y = (float)y[i], Z = (float)z[i];
        const float rho2 = X * X + Y * Y, rho = sqrtf(rho2), r = sqrtf(rho2 + Z * Z);
        const float th = m_atan2(rho, Z);
        float ph = m_atan2(Y, X);
        if (ph < 0.0f) ph += two_pi<float>();
        float fi = (r - g.r_min) * g.inv_dr, fj = th * g.inv_dth, fk = ph * g.inv_dph;
        if (!(isfinite(fi) && isfinite(fj) && isfinite(fk))) { fi = 0; fj = 0; fk = 0; }
        const int i_ = (int)fminf(fmaxf(floorf(fi), 0.0f), (float)(g.n_r - 1));
        const int j_ = (int)fminf(fmaxf(floorf(fj), 0.0f), (float)(g.n_th - 1));
        const int k_ = (int)fminf(fmaxf(floorf(fk), 0.0f), (float)(g.n_ph - 1));
        const uint32_t kk = ((uint32_t)(k_ >> g.shift) * g.nth_c + (uint32_t)(j_ >> g.shift)) * g.nr_c +
                            (uint32_t)(i_ >> g.shift);
        key[i] = kk;
        // one atomic per bin and warp: freshly injected particles all share a bin
        const unsigned grp = __match_any_sync(__activemask(), kk);
        const int leader = __ffs(grp) - 1;
        uint32_t base = 0;
        if ((int)lane == leader) base = atomicAdd(hist + kk, (uint32_t)__popc(grp));
        rank[i] = __shfl_sync(grp, base, leader) + (uint32_t)__popc(grp & ((1u << lane) - 1u));
    }
}

// exclusive scan of hist within blocks of kScanBins bins, in place; the blocks' totals to sums
constexpr int kScanBins = 1024;
__global__ void __launch_bounds__(kScanBins) scan_kernel(uint32_t *hist, int nb, uint32_t *sums)
{
    __shared__ uint32_t part[32];
    const int i = blockIdx.x * kScanBins + threadIdx.x, w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t v = i < nb ? hist[i] : 0u;
    uint32_t s = v;
    for (int off = 1; off < 32; off <<= 1) {
        const uint32_t t = __shfl_up_sync(0xffffffffu, s, off);
        if (lane >= off) s += t;
    }
    if (lane == 31) part[w] = s;
    __syncthreads();
    if (w == 0) {
        uint32_t p = part[lane];
        for (int off = 1; off < 32; off <<= 1) {
            const uint32_t t = __shfl_up_sync(0xffffffffu, p, off);
            if (lane >= off) p += t;
        }
        part[lane] = p;
    }
    __syncthreads();
    if (w > 0) s += part[w - 1];
    if (i < nb) hist[i] = s - v;
    if (threadIdx.x == kScanBins - 1) sums[blockIdx.x] = s;
}

// destination of each particle, in place of its rank; every block scans the few block sums
constexpr int kMaxScanBlocks = (1 << 18) / kScanBins;
__global__ void __launch_bounds__(kMaxScanBlocks) dest_kernel(int64_t n, const uint32_t *__restrict__ key, uint32_t *rank,
                                                              const uint32_t *__restrict__ off,
                                                              const uint32_t *__restrict__ sums, int n_sums)
{
    __shared__ uint32_t s_off[kMaxScanBlocks];
    const int t = threadIdx.x;
    const uint32_t v = t < n_sums ? sums[t] : 0u;
    s_off[t] = v;
    __syncthreads();
    for (int o = 1; o < kMaxScanBlocks; o <<= 1) {
        const uint32_t p = t >= o ? s_off[t - o] : 0u;
        __syncthreads();
        s_off[t] += p;
        __syncthreads();
    }
    s_off[t] -= v;
    __syncthreads();
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + t; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t k = key[i];
        rank[i] += off[k] + s_off[k / kScanBins];
    }
}

// all 19 double rows (11 arrays + 4 rows each of F0, F1) and 5 uint32 arrays
struct Scatter {
    const double *src_d[19];
    double *dst_d[19];
    const uint32_t *src_u[5];
    uint32_t *dst_u[5];
};

// one array per blockIdx.y (blocks of one array before those of the next): particle i to slot
// dest[i] - base
constexpr int kMovePer = 4;
__global__ void __launch_bounds__(256) move_kernel(const __grid_constant__ Scatter S, int64_t n,
                                                   const uint32_t *__restrict__ dest, uint32_t base)
{
    const int a = blockIdx.y;
    const int64_t i0 = (int64_t)blockIdx.x * (256 * kMovePer) + threadIdx.x;
    uint32_t d[kMovePer];
#pragma unroll
    for (int k = 0; k < kMovePer; ++k)
        d[k] = i0 + 256 * k < n ? dest[i0 + 256 * k] - base : 0u;
    if (a < 19) {
        const double *__restrict__ src = S.src_d[a];
        double *__restrict__ dst = S.dst_d[a];
        double v[kMovePer];
#pragma unroll
        for (int k = 0; k < kMovePer; ++k)
            v[k] = i0 + 256 * k < n ? __ldcs(src + i0 + 256 * k) : 0.0;
#pragma unroll
        for (int k = 0; k < kMovePer; ++k)
            if (i0 + 256 * k < n) dst[d[k]] = v[k];
    } else {
        const uint32_t *__restrict__ src = S.src_u[a - 19];
        uint32_t *__restrict__ dst = S.dst_u[a - 19];
        uint32_t v[kMovePer];
#pragma unroll
        for (int k = 0; k < kMovePer; ++k)
            v[k] = i0 + 256 * k < n ? src[i0 + 256 * k] : 0u;
#pragma unroll
        for (int k = 0; k < kMovePer; ++k)
            if (i0 + 256 * k < n) dst[d[k]] = v[k];
    }
}

void move_arrays(const Scatter &S, int64_t n, const uint32_t *dest, uint32_t base, cudaStream_t s)
{
    const int64_t per = 256 * kMovePer;
    move_kernel<<<dim3((unsigned)((n + per - 1) / per), 24), 256, 0, s>>>(S, n, dest, base);
}

Scatter make_scatter(const StateDev &st, const StateDev &alt)
{
    Scatter S;
    const double *sd[11] = {st.x, st.y, st.z, st.u, st.mub, st.vpar, st.s_rem, st.h_prev,
                            st.t_birth, st.u_inj, st.mub_inj};
    double *dd[11] = {alt.x, alt.y, alt.z, alt.u, alt.mub, alt.vpar, alt.s_rem, alt.h_prev,
                      alt.t_birth, alt.u_inj, alt.mub_inj};
    for (int a = 0; a < 11; ++a) {
        S.src_d[a] = sd[a];
        S.dst_d[a] = dd[a];
    }
    for (int r = 0; r < 4; ++r) {
        S.src_d[11 + r] = st.F0 + r * st.cap;
        S.dst_d[11 + r] = alt.F0 + r * st.cap;
        S.src_d[15 + r] = st.F1 + r * st.cap;
        S.dst_d[15 + r] = alt.F1 + r * st.cap;
    }
    const uint32_t *su[5] = {st.id, st.ens, st.event, st.ncoll, st.flags};
    uint32_t *du[5] = {alt.id, alt.ens, alt.event, alt.ncoll, alt.flags};
    for (int a = 0; a < 5; ++a) {
        S.src_u[a] = su[a];
        S.dst_u[a] = du[a];
    }
    return S;
}

void free_alt(StateDev &s)
{
    double *d[] = {s.x, s.y, s.z, s.u, s.mub, s.vpar, s.s_rem, s.h_prev, s.t_birth, s.u_inj, s.mub_inj, s.F0, s.F1};
    for (double *p : d)
        if (p) cudaFree(p);
    uint32_t *u[] = {s.id, s.ens, s.event, s.ncoll, s.flags};
    for (uint32_t *p : u)
        if (p) cudaFree(p);
    s = StateDev{};
}

cudaError_t alloc_alt(StateDev &s, int64_t cap)
{
    double **d[] = {&s.x, &s.y, &s.z, &s.u, &s.mub, &s.vpar, &s.s_rem, &s.h_prev, &s.t_birth, &s.u_inj, &s.mub_inj};
    for (double **p : d) {
        const cudaError_t e = cudaMalloc(p, (size_t)cap * 8);
        if (e != cudaSuccess) return e;
    }
    cudaError_t e = cudaMalloc(&s.F0, (size_t)cap * 32);
    if (e != cudaSuccess) return e;
    e = cudaMalloc(&s.F1, (size_t)cap * 32);
    if (e != cudaSuccess) return e;
    uint32_t **u[] = {&s.id, &s.ens, &s.event, &s.ncoll, &s.flags};
    for (uint32_t **p : u) {
        e = cudaMalloc(p, (size_t)cap * 4);
        if (e != cudaSuccess) return e;
    }
    s.cap = cap;
    return cudaSuccess;
}

cudaError_t ensure_alt(SortWork &w, int64_t cap)
{
    if (w.cap == cap) return cudaSuccess;
    free_alt(w.alt);
    if (w.key) cudaFree(w.key);
    if (w.rank) cudaFree(w.rank);
    w.key = w.rank = nullptr;
    w.cap = 0;
    cudaError_t e;
    if ((e = alloc_alt(w.alt, cap)) != cudaSuccess) { free_alt(w.alt); return e; }
    if ((e = cudaMalloc(&w.key, (size_t)cap * 4)) != cudaSuccess) return e;
    if ((e = cudaMalloc(&w.rank, (size_t)cap * 4)) != cudaSuccess) return e;
    w.cap = cap;
    return cudaSuccess;
}

int grid_for(int64_t n, int block) { return (int)std::min<int64_t>((n + block - 1) / block, 152 * 16); }

} // namespace

void sort_free(SortWork &w)
{
    free_alt(w.alt);
    if (w.key) cudaFree(w.key);
    if (w.rank) cudaFree(w.rank);
    if (w.hist) cudaFree(w.hist);
    w = SortWork{};
}

cudaError_t unpermute_to_alt(SortWork &w, const StateDev &st, uint32_t id_lo, cudaStream_t s)
{
    const int64_t n = st.n;
    if (n == 0) return cudaSuccess;
    cudaError_t e;
    if ((e = ensure_alt(w, st.cap)) != cudaSuccess) return e;
    move_arrays(make_scatter(st, w.alt), n, st.id, id_lo, s);
    return cudaGetLastError();
}

namespace {
KeyGeom key_geom(const GridHost &g, int64_t *nbins)
{
    KeyGeom kg;
    kg.r_min = (float)(g.r_min);
    kg.inv_dr = (float)(1.0 / g.dr);
    kg.inv_dth = (float)(1.0 / g.dth);
    kg.inv_dph = (float)(1.0 / g.dph);
    kg.n_r = g.n_r;
    kg.n_th = g.n_th;
    kg.n_ph = g.n_ph;
    kg.shift = 0;
    auto bins = [&](int sh) {
        return (int64_t)(((g.n_r - 1) >> sh) + 1) * (((g.n_th - 1) >> sh) + 1) * (((g.n_ph - 1) >> sh) + 1);
    };
    while (bins(kg.shift) > (1 << 18)) ++kg.shift;
    kg.nr_c = ((g.n_r - 1) >> kg.shift) + 1;
    kg.nth_c = ((g.n_th - 1) >> kg.shift) + 1;
    kg.nph_c = ((g.n_ph - 1) >> kg.shift) + 1;
    *nbins = bins(kg.shift);
    return kg;
}

cudaError_t ensure_hist(SortWork &w, int64_t nb)
{
    if (w.nbins_cap >= nb) return cudaSuccess;
    if (w.hist) cudaFree(w.hist);
    w.hist = nullptr;
    w.nbins_cap = 0;
    const cudaError_t e = cudaMalloc(&w.hist, (size_t)(nb + kMaxScanBlocks) * 4); // counts, block sums
    if (e == cudaSuccess) w.nbins_cap = nb;
    return e;
}
} // namespace

cudaError_t alloc_state(StateDev &s, int64_t cap) { return alloc_alt(s, cap); }

cudaError_t sort_preload()
{
    cudaFuncAttributes a;
    cudaError_t e = cudaFuncGetAttributes(&a, key_kernel);
    if (e == cudaSuccess) e = cudaFuncGetAttributes(&a, scan_kernel);
    if (e == cudaSuccess) e = cudaFuncGetAttributes(&a, dest_kernel);
    if (e == cudaSuccess) e = cudaFuncGetAttributes(&a, move_kernel);
    return e;
}
void free_state_arrays(StateDev &s) { free_alt(s); }

cudaError_t sort_reserve(SortWork &w, const StateDev &st, const GridHost &g)
{
    int64_t nb = 0;
    key_geom(g, &nb);
    cudaError_t e = ensure_alt(w, st.cap);
    if (e != cudaSuccess) return e;
    return ensure_hist(w, nb);
}

cudaError_t sort_by_cell(SortWork &w, StateDev &st, const GridHost &g, int n_ens, cudaStream_t s)
{
    (void)n_ens;
    const int64_t n = st.n;
    if (n < 2) return cudaSuccess;
    cudaGetLastError(); // report this sort's errors only
    int64_t nb = 0;
    const KeyGeom kg = key_geom(g, &nb);
    cudaError_t e;
    if ((e = ensure_alt(w, st.cap)) != cudaSuccess) return e;
    if ((e = ensure_hist(w, nb)) != cudaSuccess) return e;
    if ((e = cudaMemsetAsync(w.hist, 0, (size_t)nb * 4, s)) != cudaSuccess) return e;
    const int grid = grid_for(n, 256);
    key_kernel<<<grid, 256, 0, s>>>(st.x, st.y, st.z, n, kg, w.key, w.rank, w.hist);
    const int n_sums = (int)((nb + kScanBins - 1) / kScanBins);
    uint32_t *sums = w.hist + nb;
    scan_kernel<<<n_sums, kScanBins, 0, s>>>(w.hist, (int)nb, sums);
    dest_kernel<<<(unsigned)std::min<int64_t>((n + kMaxScanBlocks - 1) / kMaxScanBlocks, 152 * 8), kMaxScanBlocks, 0, s>>>(
        n, w.key, w.rank, w.hist, sums, n_sums);
    move_arrays(make_scatter(st, w.alt), n, w.rank, 0u, s);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    // swap: the sorted copy becomes the state
    StateDev old = st;
    StateDev nw = w.alt;
    nw.n = old.n;
    nw.cap = old.cap;
    old.n = 0;
    w.alt = old;
    st = nw;
    return cudaSuccess;
}

} // namespace gcp
