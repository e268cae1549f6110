// Saturated nuclei (8Be with relativistic operators: all 12 u and all 12 d
// quark states taken): C_c(x) = coef_c det S(x)^2 (Sec. 8; plan.h), one 12 x 12
// determinant per site instead of the recursion's 448,496,928 complex
// multiply-adds. Gaussian elimination with partial pivoting in FP64 for both
// arithmetics: 2.3 K FP64 multiply-adds per site are too few for FP32 to pay.
//
// Half a warp owns a site, lane r < 12 holds row r in registers. A step picks
// the pivot row by the largest |re| + |im| (compared on the high words), sends
// it to the other rows by shuffles and eliminates; rows stay where they are,
// the permutation's sign is counted. The kernel is bound by the FP64 units (a
// warp's FP64 instruction takes one of the SM's four for 64 cycles) through
// 12 dependent steps. Measured on GB300 against the recursion, whole calls: 64
// sites FP64 198.0 ms -> 43 us, 512 sites mixed 156.1 ms -> 57 us (the kernel
// 36 us of it).
#pragma once

#include "small_kernel.cuh"

namespace mbc {

// Sites per CTA and tile: the warps of an SM share its FP64 unit, so lattices
// of few sites take one warp per CTA to reach every SM.
constexpr int kSatWide = 8, kSatNarrow = 2;

// det of the 12 x 12 matrix whose row (lane & 15) this lane holds
__device__ __forceinline__ double2 det12(double2 (&a)[12]) {
    const int row = threadIdx.x & 15;
    const unsigned half = 0xffffu << (threadIdx.x & 16);
    unsigned left = 0xfffu;  // rows not yet used as pivots
    unsigned odd = 0;
    double2 det = make_double2(1.0, 0.0);
#pragma unroll
    for (int k = 0; k < 12; ++k) {
        // +1 keeps zero rows above the used ones; NaN compares above all
        const uint32_t key =
            (left >> row & 1u) ? (uint32_t)__double2hiint(fabs(a[k].x) + fabs(a[k].y)) + 1u : 0u;
        const uint32_t best = __reduce_max_sync(half, key);
        const int p = __ffs((__ballot_sync(half, key == best) >> (threadIdx.x & 16)) & 0xffffu) - 1;
        odd ^= __popc(left & ((1u << p) - 1u)) & 1u;
        left &= ~(1u << p);
        const double2 piv = make_double2(__shfl_sync(half, a[k].x, p, 16), __shfl_sync(half, a[k].y, p, 16));
        det = cmul(det, piv);
        // factor = a[k] / piv; pivots whose square would overflow or vanish are
        // scaled first (with the column) by their exponent. A zero pivot has a
        // zero column below it and nothing to eliminate
        const double big = fmax(fabs(piv.x), fabs(piv.y));
        double2 num = a[k], den = piv;
        if (!(big > 0x1p-480 && big < 0x1p480)) {
            const int e = big > 0.0 ? -ilogb(big) : 0;
            num = make_double2(scalbn(num.x, e), scalbn(num.y, e));
            den = make_double2(scalbn(den.x, e), scalbn(den.y, e));
        }
        const double inv = big == 0.0 ? 0.0 : 1.0 / __fma_rn(den.x, den.x, den.y * den.y);
        const double2 f = make_double2(__fma_rn(num.x, den.x, num.y * den.y) * inv,
                                       __fma_rn(num.y, den.x, -num.x * den.y) * inv);
#pragma unroll
        for (int j = k + 1; j < 12; ++j) {
            const double2 q = make_double2(__shfl_sync(half, a[j].x, p, 16), __shfl_sync(half, a[j].y, p, 16));
            if (left >> row & 1u) a[j] = cfms(f, q, a[j]);
        }
    }
    return odd ? make_double2(-det.x, -det.y) : det;
}

// partial[tile][mom][comp]: phase-weighted sums over the tile's sites in a
// fixed order, scaled by the component's coefficient
template <int kSatSites>
__global__ void __launch_bounds__(16 * kSatSites)
    k_saturated(FieldDesc F, MomDesc M, const double *__restrict__ coef, int n_comp, int tiles_per_slab,
                double2 *__restrict__ partial) {
    __shared__ double2 d2[kSatSites], sum[kMaxMom];
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
    const double2 d = det12(a);
    if (row == 0) d2[s] = live ? cmul(d, d) : make_double2(0.0, 0.0);
    __syncthreads();
    for (int q = threadIdx.x; q < M.n_mom; q += blockDim.x) {
        double re = 0.0, im = 0.0;
        for (int w = 0; w < kSatSites && site0 + w < v3; ++w) {
            const int site = site0 + w;
            const double2 ph = mom_phase(M.mom[q], site % F.lx, (site / F.lx) % F.ly, site / (F.lx * F.ly), F.lx, F.ly,
                                         F.lz);
            re = __fma_rn(ph.x, d2[w].x, __fma_rn(-ph.y, d2[w].y, re));
            im = __fma_rn(ph.x, d2[w].y, __fma_rn(ph.y, d2[w].x, im));
        }
        sum[q] = make_double2(re, im);
    }
    __syncthreads();
    for (int o = threadIdx.x; o < M.n_mom * n_comp; o += blockDim.x) {
        const double c = __ldg(coef + o % n_comp);
        partial[tile * (int64_t)(M.n_mom * n_comp) + o] = make_double2(c * sum[o / n_comp].x, c * sum[o / n_comp].y);
    }
}

}  // namespace mbc
