// Saturated nuclei (8Be with relativistic operators: all 12 u and all 12 d
// quark states taken): C_c(x) = coef_c det S(x)^2 (Sec. 8; plan.h), one 12 x 12
// determinant per site instead of the recursion's 448,496,928 complex
// multiply-adds. Gaussian elimination with partial pivoting in FP64 for both
// arithmetics: 2.3 K FP64 multiply-adds per site are too few for FP32 to pay.
//
// Half a warp owns a site, lane r < 12 holds row r in registers. A step picks
// the pivot row by the largest |re| + |im| (compared on the high words), sends
// it to the other rows by shuffles and eliminates; rows stay where they are (the
// permutation's sign squares away). The kernel is bound by the FP64 units (a
// warp's FP64 instruction takes one of the SM's four for 64 cycles) through
// 12 dependent steps. Measured on GB300 against the recursion, whole calls: 64
// sites FP64 198.0 ms -> 27 us, 512 sites mixed 156.1 ms -> 55 us (host and launches
// more than half of both), 16^3 sites FP64 86 us, with 4 momenta 91.
#pragma once

#include <cooperative_groups.h>

#include "small_kernel.cuh"

namespace mbc {

// Sites per CTA and tile.
constexpr int kSatSites = 8;

// a / piv; pivots whose square would overflow or vanish are scaled first (with a)
// by their exponent. A zero pivot has a zero column below it and nothing to
// eliminate.
__device__ __forceinline__ double2 pivot_factor(double2 a, double2 piv) {
    const double big = fmax(fabs(piv.x), fabs(piv.y));
    if (!(big > 0x1p-480 && big < 0x1p480)) {
        const int e = big > 0.0 ? -ilogb(big) : 0;
        a = make_double2(scalbn(a.x, e), scalbn(a.y, e));
        piv = make_double2(scalbn(piv.x, e), scalbn(piv.y, e));
    }
    const double inv = big == 0.0 ? 0.0 : 1.0 / __fma_rn(piv.x, piv.x, piv.y * piv.y);
    return make_double2(__fma_rn(a.x, piv.x, a.y * piv.y) * inv, __fma_rn(a.y, piv.x, -a.x * piv.y) * inv);
}

// det, up to its sign, of the 12 x 12 matrix whose row (lane & 15) this lane holds.
// The pivots are multiplied in the order of k_saturated_few's tree.
__device__ __forceinline__ double2 det12(double2 (&a)[12]) {
    const int row = threadIdx.x & 15;
    const unsigned half = 0xffffu << (threadIdx.x & 16);
    unsigned left = 0xfffu;  // rows not yet used as pivots
#pragma unroll
    for (int k = 0; k < 12; ++k) {
        // +1 keeps zero rows above the used ones; NaN compares above all
        const uint32_t key =
            (left >> row & 1u) ? (uint32_t)__double2hiint(fabs(a[k].x) + fabs(a[k].y)) + 1u : 0u;
        const uint32_t best = __reduce_max_sync(half, key);
        const int p = __ffs((__ballot_sync(half, key == best) >> (threadIdx.x & 16)) & 0xffffu) - 1;
        left &= ~(1u << p);
        const double2 piv = make_double2(__shfl_sync(half, a[k].x, p, 16), __shfl_sync(half, a[k].y, p, 16));
        const double2 f = pivot_factor(a[k], piv);
        a[k] = piv;  // the column is done with: its place keeps the pivot
#pragma unroll
        for (int j = k + 1; j < 12; ++j) {
            const double2 q = make_double2(__shfl_sync(half, a[j].x, p, 16), __shfl_sync(half, a[j].y, p, 16));
            if (left >> row & 1u) a[j] = cfms(f, q, a[j]);
        }
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) a[i] = cmul(cmul(a[i], a[i + 8]), a[i + 4]);
    return cmul(cmul(a[0], a[2]), cmul(a[1], a[3]));
}

// What the sums over a tile's sites read: squared determinants and phases.
struct SatTile {
    double2 d2[kSatSites], ph[kSatSites][kMaxMom], sum[kMaxMom];
};
__device__ __forceinline__ double2 sat_phase(const FieldDesc &F, const MomDesc &M, int site, int q) {
    return mom_phase(M.mom[q], site % F.lx, (site / F.lx) % F.ly, site / (F.lx * F.ly), F.lx, F.ly, F.lz);
}

// partial[tile][mom][comp]: phase-weighted sums over the tile's sites in a fixed
// tree, scaled by the component's coefficient; a lane takes a real or imaginary part
__device__ __forceinline__ void saturated_sums(SatTile &T, const FieldDesc &F, const MomDesc &M, const double *coef,
                                               int n_comp, int64_t tile, int site0, double2 *partial) {
    const int n = min(kSatSites, F.lx * F.ly * F.lz - site0);
    for (int i = threadIdx.x; i < 2 * M.n_mom; i += blockDim.x) {
        const bool im = i & 1;
        double t[kSatSites];
#pragma unroll
        for (int w = 0; w < kSatSites; ++w) {
            const double2 d = T.d2[w], ph = T.ph[w][i >> 1];
            t[w] = w < n ? __fma_rn(ph.x, im ? d.y : d.x, (im ? ph.y : -ph.y) * (im ? d.x : d.y)) : 0.0;
        }
#pragma unroll
        for (int off = 1; off < kSatSites; off *= 2)
#pragma unroll
            for (int w = 0; w < kSatSites; w += 2 * off) t[w] += t[w + off];
        reinterpret_cast<double *>(T.sum)[i] = t[0];
    }
    __syncthreads();
    for (int o = threadIdx.x; o < M.n_mom * n_comp; o += blockDim.x) {
        const double c = __ldg(coef + o % n_comp);
        partial[tile * (int64_t)(M.n_mom * n_comp) + o] = make_double2(c * T.sum[o / n_comp].x, c * T.sum[o / n_comp].y);
    }
}

__global__ void __launch_bounds__(16 * kSatSites)
    k_saturated(FieldDesc F, MomDesc M, const double *__restrict__ coef, int n_comp, int tiles_per_slab,
                double2 *__restrict__ partial) {
    __shared__ SatTile T;
    const int64_t tile = blockIdx.x, slab = tile / tiles_per_slab;
    const int site0 = (int)(tile % tiles_per_slab) * kSatSites, v3 = F.lx * F.ly * F.lz;
    const int s = threadIdx.x >> 4, row = threadIdx.x & 15;
    const bool live = site0 + s < v3;
    double2 a[12];
#pragma unroll
    for (int j = 0; j < 12; ++j) a[j] = make_double2(0.0, 0.0);
    if (live && row < 12) {
        const int64_t base = slab / F.n_t * F.stride_cfg + (F.t0 + slab % F.n_t) * F.stride_t + (int64_t)(site0 + s) * 144;
#pragma unroll
        for (int j = 0; j < 12; ++j) a[j] = load_prop(F, base, row * 12 + j);
    }
    // phases: an FP64 sine and cosine each, so every thread takes some
    for (int o = threadIdx.x; o < kSatSites * M.n_mom; o += blockDim.x)
        if (site0 + o / M.n_mom < v3) T.ph[o / M.n_mom][o % M.n_mom] = sat_phase(F, M, site0 + o / M.n_mom, o % M.n_mom);
    const double2 d = det12(a);
    if (row == 0) T.d2[s] = cmul(d, d);
    __syncthreads();
    saturated_sums(T, F, M, coef, n_comp, tile, site0, partial);
}

// The same elimination with a CTA of four warps per site, for lattices of few
// sites: a warp's FP64 instructions run on one of the SM's four FP64 units, so
// one warp per site leaves three idle. Lanes are rows, twice; warp w holds columns
// w, w + 4 (upper half) and w + 8. The warp that owns a step's column finds the
// pivot and writes the rows' factors to shared memory; every warp then fetches its
// columns' pivot elements by shuffles and eliminates. 64 sites: 17 us, one warp
// for two sites 30. The CTAs of a tile are a cluster (sat_cluster of them) whose first
// one sums the sites: the operations and their order are k_saturated's, and so are
// the bits.
inline int sat_cluster(int64_t v3) { return v3 > 4 ? kSatSites : v3 > 2 ? 4 : v3 > 1 ? 2 : 1; }
__global__ void __launch_bounds__(128)
    k_saturated_few(FieldDesc F, MomDesc M, const double *__restrict__ coef, int n_comp, int tiles_per_slab,
                    double2 *__restrict__ partial) {
    __shared__ SatTile T;
    __shared__ double2 fac[2][12], pivots[12];
    __shared__ int prow[2];
    const cooperative_groups::cluster_group cluster = cooperative_groups::this_cluster();
    const int v3 = F.lx * F.ly * F.lz;
    const int ctas = (int)cluster.num_blocks(), in_tile = (int)cluster.block_rank();
    const int64_t tile = blockIdx.x / ctas, slab = tile / tiles_per_slab;
    const int site0 = (int)(tile % tiles_per_slab) * kSatSites, site = site0 + in_tile;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, half = lane >> 4, row = lane & 15;
    double2 a[2] = {make_double2(0.0, 0.0), make_double2(0.0, 0.0)};  // columns w + 4 half, w + 8 (lower half)
    const bool live = site < v3;  // a tile's last CTAs may have no site
    if (live && row < 12) {
        const int64_t base = slab / F.n_t * F.stride_cfg + (F.t0 + slab % F.n_t) * F.stride_t + (int64_t)site * 144;
        a[0] = load_prop(F, base, row * 12 + w + 4 * half);
        if (half == 0) a[1] = load_prop(F, base, row * 12 + w + 8);
    }
    unsigned left = 0xfffu;
#pragma unroll
    for (int k = 0; k < 12; ++k) {
        if (!live) break;
        const int h = (k >> 2) & 1, q = k >> 3;  // column k: warp k % 4, half h, register q
        if (w == (k & 3) && half == h) {
            const unsigned mask = 0xffffu << (16 * h);
            const uint32_t key =
                (left >> row & 1u) ? (uint32_t)__double2hiint(fabs(a[q].x) + fabs(a[q].y)) + 1u : 0u;
            const uint32_t best = __reduce_max_sync(mask, key);
            const int p = __ffs((__ballot_sync(mask, key == best) >> (16 * h)) & 0xffffu) - 1;
            const double2 piv = make_double2(__shfl_sync(mask, a[q].x, p, 16), __shfl_sync(mask, a[q].y, p, 16));
            const double2 f = pivot_factor(a[q], piv);
            if (row < 12) fac[k & 1][row] = (left >> row & 1u) && row != p ? f : make_double2(0.0, 0.0);
            if (row == 0) {
                prow[k & 1] = p;
                pivots[k] = piv;
            }
        }
        __syncthreads();  // double-buffered: a step's readers are done before the next but one writes
        const int p = prow[k & 1];
        left &= ~(1u << p);
        const double2 f = row < 12 ? fac[k & 1][row] : make_double2(0.0, 0.0);
#pragma unroll
        for (int g = 0; g < 2; ++g) {
            if (g == 0 ? w + 4 <= k : w + 8 <= k) continue;  // no column of this group is left
            const double2 x = make_double2(__shfl_sync(0xffffffffu, a[g].x, p, 16), __shfl_sync(0xffffffffu, a[g].y, p, 16));
            if (w + 4 * half + 8 * g > k && (left >> row & 1u)) a[g] = cfms(f, x, a[g]);
        }
    }
    cluster.sync();  // the first CTA has started (every pivot is written by now)
    SatTile *first = cluster.map_shared_rank(&T, 0);
    if (w > 0 && live) {
        for (int q = threadIdx.x - 32; q < M.n_mom; q += 96) first->ph[in_tile][q] = sat_phase(F, M, site, q);
    } else if (live) {  // product of the pivots, in a fixed tree
        double2 d = lane < 12 ? pivots[lane] : make_double2(1.0, 0.0);
        for (int off = 8; off > 0; off >>= 1) {
            const double2 o = make_double2(__shfl_xor_sync(0xffffffffu, d.x, off), __shfl_xor_sync(0xffffffffu, d.y, off));
            if (off < 8 || lane < 4) d = cmul(d, o);  // four pivots have no partner eight further
        }
        if (lane == 0) first->d2[in_tile] = cmul(d, d);
    }
    cluster.sync();  // the tile's determinants and phases are in the first CTA
    if (in_tile == 0) saturated_sums(T, F, M, coef, n_comp, tile, site0, partial);
}

}  // namespace mbc
