// Minor form of the nonrelativistic nuclei (plan.h), lanes are sites: a CTA owns a
// tile of 32 sites and keeps every minor as a row of 32 lanes in shared memory
// ([entry][lane], conflict-free). The warps split the outputs of an order; an
// output's operation words are read by all lanes at once (7 KB, L1), its two to
// six products unrolled. The next tile's propagators are in flight while one is
// contracted.
//
// FP64 is bound by its pipe (2.0 K complex multiply-adds per site for 3He + 4He,
// 80 % of it on 16^3 x 32: 2.14 ms); one warp per site (k_small, 2.69 ms) keeps the
// lattices that have fewer tiles than SMs. Mixed (0.48 ms; 0.86 with k_small_ls) is
// bound by its barriers and FP32 issue (54 %). u and d share their minors, so a
// rounding counts in both factors; where an operand is a propagator entry the
// mixed form therefore takes its low word along, and second-order minors use exact
// products (errors against FP64 below the recursion's).
#pragma once

#include "small_ls_kernel.cuh"

namespace mbc {

// warps per CTA: one CTA per SM in FP64 (190 KB for 3He), two in mixed precision
__host__ __device__ constexpr int minor_warps(bool mixed) { return mixed ? 16 : 24; }
constexpr int kMinorParts = 32;  // partial sums of the runs (kMaxMinorRuns at least)

// low word of an FP64 value scaled by 2^e: d 2^e - f64_scaled_to_f32(d, e), to FP32
__device__ __forceinline__ float f64_scaled_low(double d, int e) {
    const uint32_t hi = (uint32_t)__double2hiint(d), lo = (uint32_t)__double2loint(d);
    const int eb = (int)((hi >> 20) & 0x7ffu), ef = eb - 1023 + e + 127;
    if (eb == 0 || ef <= 52) return 0.f;  // below FP32's range with the 52 bits' weight
    const uint32_t top = ((hi & 0xfffffu) << 3) | (lo >> 29), rem = lo & 0x1fffffffu;
    const bool up = rem > 0x10000000u || (rem == 0x10000000u && (top & 1u));
    const float r = (float)((int)rem - (up ? 0x20000000 : 0));  // units of 2^(ef - 127 - 52)
    const float v = r * __int_as_float((ef - 52) << 23);
    return (hi & 0x80000000u) ? -v : v;
}

// Sums of products per output. Mixed: compensated FP32; xs(): x has a low word,
// ss(): both have and the products are exact.
struct MinorAcc64 {
    FP64Traits::Acc a;
    __device__ __forceinline__ void zero() { a.zero(); }
    __device__ __forceinline__ void plain(double2 x, double2 y, uint32_t neg) { a.fma(x, y, neg); }
    __device__ __forceinline__ double2 store() const { return a.store(); }
};
struct MinorAccMx {
    MixedTraits::Acc a;
    __device__ __forceinline__ void zero() { a.zero(); }
    __device__ __forceinline__ void plain(float2 x, float2 y, uint32_t neg) { a.fma(x, y, neg); }
    __device__ __forceinline__ static void flip(float2 &x, uint32_t neg) {
        x.x = __int_as_float(__float_as_int(x.x) ^ (int)neg);
        x.y = __int_as_float(__float_as_int(x.y) ^ (int)neg);
    }
    // n += x y
    __device__ __forceinline__ void low(float2 x, float2 y) {
        a.n = f2_fma(f2_pack(x.x, x.x), f2_pack(y.x, y.y), a.n);
        a.n = f2_fma(f2_pack(-x.y, x.y), f2_pack(y.y, y.x), a.n);
    }
    __device__ __forceinline__ void xs(float2 x, float2 xl, float2 y, uint32_t neg) {
        flip(xl, neg);
        a.fma(x, y, neg);
        low(xl, y);
    }
    __device__ __forceinline__ void ss(float2 x, float2 xl, float2 y, float2 yl, uint32_t neg) {
        flip(x, neg);
        flip(xl, neg);
        const uint64_t xr = f2_pack(x.x, x.x), xi = f2_pack(-x.y, x.y), y1 = f2_pack(y.x, y.y), y2 = f2_pack(y.y, y.x);
        const uint64_t p1 = f2_mul(xr, y1), p2 = f2_mul(xi, y2);
        const uint64_t e = f2_add(f2_fma(xr, y1, f2_neg(p1)), f2_fma(xi, y2, f2_neg(p2)));
        f2_kahan(a.s, a.n, p1);
        f2_kahan(a.s, a.n, p2);
        a.n = f2_add(a.n, e);
        low(xl, y);
        low(x, yl);
    }
    __device__ __forceinline__ float2 store() const { return a.store(); }
};

template <class Tr>
struct MinorRows {
    using V = typename Tr::V;
    static constexpr bool kMx = sizeof(V) == 8;
    static constexpr int kRow = 32 * (int)sizeof(V);  // bytes
    static constexpr int kWarps = minor_warps(kMx);
    using Acc = std::conditional_t<kMx, MinorAccMx, MinorAcc64>;
};

// One order: outputs z = warp, warp + kWarps, ...; K products each. S: the
// operands' x rows (SX) and y rows (SY) are the tile, whose low words lie low_off
// bytes further (mixed).
template <class Tr, int K, bool SX, bool SY>
__device__ __forceinline__ void minor_step(const unsigned char *X, const unsigned char *Y, unsigned char *Z,
                                           const uint32_t *__restrict__ ops, int n_z, int low_off, int warp) {
    using M = MinorRows<Tr>;
    using V = typename Tr::V;
    for (int z = warp; z < n_z; z += M::kWarps) {
        uint32_t op[K];
#pragma unroll
        for (int j = 0; j < K; ++j) op[j] = __ldg(ops + z * K + j);
        typename M::Acc acc;
        acc.zero();
#pragma unroll
        for (int j = 0; j < K; ++j) {
            const unsigned char *xp = X + ((op[j] >> 8 & 0xffu) * M::kRow), *yp = Y + ((op[j] >> 24) * M::kRow);
            const uint32_t neg = op[j] << 31;
            const V x = *reinterpret_cast<const V *>(xp), y = *reinterpret_cast<const V *>(yp);
            if constexpr (M::kMx && SX && SY)
                acc.ss(x, *reinterpret_cast<const V *>(xp + low_off), y, *reinterpret_cast<const V *>(yp + low_off), neg);
            else if constexpr (M::kMx && SX)
                acc.xs(x, *reinterpret_cast<const V *>(xp + low_off), y, neg);
            else
                acc.plain(x, y, neg);
        }
        *reinterpret_cast<V *>(Z + z * M::kRow) = acc.store();
    }
}

template <class Tr>
__global__ void __launch_bounds__(32 * MinorRows<Tr>::kWarps, MinorRows<Tr>::kMx ? 2 : 1)
    k_minors(const __grid_constant__ SmallBatch B, FieldDesc F, MomDesc M, const double2 *__restrict__ phase,
             double2 *partial_base) {
    using T = MinorRows<Tr>;
    using V = typename Tr::V;
    constexpr bool kMx = T::kMx;
    constexpr int kMinorWarps = T::kWarps;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ int sexp_s[2][32];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int V3 = F.lx * F.ly * F.lz;
    unsigned char *R = smem_raw + lane * sizeof(V);                      // row e of this lane: R + e * kRow
    const int low_off = B.site_stride * T::kRow;                         // mixed: the tile's low words (36 rows); s_off = 0
    constexpr int NE = (36 + kMinorWarps - 1) / kMinorWarps;             // tile entries per warp
    double2 in[NE];
    auto fetch = [&](int64_t tile) {
        const int64_t slab = tile / B.tiles_per_slab;
        const int site = (int)(tile % B.tiles_per_slab) * 32 + lane;
        const int64_t base = slab / F.n_t * F.stride_cfg + (F.t0 + slab % F.n_t) * F.stride_t + (int64_t)site * 144;
#pragma unroll
        for (int q = 0; q < NE; ++q) {
            const int e = warp + q * kMinorWarps;
            in[q] = e < 36 && tile < B.total_items && site < V3 ? load_prop(F, base, e / 6 * 12 + e % 6) : make_double2(0, 0);
        }
    };
    if (threadIdx.x < 64) sexp_s[threadIdx.x >> 5][lane] = -100000;
    fetch(blockIdx.x);
    __syncthreads();
    int buf = 0;
    for (int64_t tile = blockIdx.x; tile < B.total_items; tile += gridDim.x, buf ^= 1) {
        // 1. the tile's propagators; mixed: scaled per site by the exact power of
        // two that brings the largest entry into [1, 2)
        int se = 0;
        if constexpr (kMx) {
            int emax = -100000;
#pragma unroll
            for (int q = 0; q < NE; ++q) emax = max(emax, max(f64_exponent(in[q].x), f64_exponent(in[q].y)));
            atomicMax(&sexp_s[buf][lane], emax);
            __syncthreads();
            emax = sexp_s[buf][lane];
            se = emax == -100000 ? 0 : -emax;
        }
#pragma unroll
        for (int q = 0; q < NE; ++q) {
            const int e = warp + q * kMinorWarps;
            if (e >= 36) continue;
            if constexpr (kMx) {
                *reinterpret_cast<float2 *>(R + e * T::kRow) = make_float2(f64_scaled_to_f32(in[q].x, se), f64_scaled_to_f32(in[q].y, se));
                *reinterpret_cast<float2 *>(R + e * T::kRow + low_off) =
                    make_float2(f64_scaled_low(in[q].x, se), f64_scaled_low(in[q].y, se));
            } else {
                *reinterpret_cast<double2 *>(R + e * T::kRow) = in[q];
            }
        }
        fetch(tile + gridDim.x);
        __syncthreads();
        if (kMx && threadIdx.x < 32) sexp_s[buf ^ 1][lane] = -100000;  // read by no one until the next tile
        const int site = (int)(tile % B.tiles_per_slab) * 32 + lane;
        const bool live = site < V3;
        for (int li = 0; li < B.n_lists; ++li) {
            const SmallPlan &P = B.plan[li];
            unsigned char *parts = R + P.part_off * T::kRow;  // [kMinorParts] sums, mixed two rows each
            // 2. the minors, order by order
            for (int m = 0; m < P.n_steps; ++m) {
                const SmallStepDesc &d = P.step[m];
                const unsigned char *X = R + d.x_off * T::kRow, *Y = R + d.y_off * T::kRow;
                unsigned char *Z = R + d.z_off * T::kRow;
                const uint32_t *ops = P.zops + d.zop_off;
                // k tells the order: 2 from two tile rows; 3 and 5 from a tile row
                // and the next lower order; 6 products make order 4 (two second-
                // order minors) or order 6 (a tile row and order 5)
                switch (d.k) {
                case 2: minor_step<Tr, 2, true, true>(X, Y, Z, ops, d.n_z, low_off, warp); break;
                case 3: minor_step<Tr, 3, true, false>(X, Y, Z, ops, d.n_z, low_off, warp); break;
                case 5: minor_step<Tr, 5, true, false>(X, Y, Z, ops, d.n_z, low_off, warp); break;
                default:
                    if (d.x_off == P.s_off)
                        minor_step<Tr, 6, true, false>(X, Y, Z, ops, d.n_z, low_off, warp);
                    else
                        minor_step<Tr, 6, false, false>(X, Y, Z, ops, d.n_z, low_off, warp);
                }
                __syncthreads();
            }
            // 3. sums of products of two minors, each run in several parts
            const int n_runs = P.run_off[P.n_comp], per = n_runs > 0 ? max(1, kMinorParts / n_runs) : 1;
            for (int u = warp; u < n_runs * per; u += kMinorWarps) {
                const int r = u / per, part = u % per, t0 = __ldg(P.term_off + r), nt = __ldg(P.term_off + r + 1) - t0;
                typename T::Acc acc;
                acc.zero();
                for (int e = t0 + part * nt / per; e < t0 + (part + 1) * nt / per; ++e) {
                    const uint32_t op = __ldg(P.terms + e);
                    acc.plain(*reinterpret_cast<const V *>(R + (op & 0xffffu) * T::kRow),
                              *reinterpret_cast<const V *>(R + (op >> 16 & 0x7fffu) * T::kRow), op & 0x80000000u);
                }
                if constexpr (kMx) {
                    *reinterpret_cast<float2 *>(parts + 2 * u * T::kRow) = f2_unpack(acc.a.s);
                    *reinterpret_cast<float2 *>(parts + (2 * u + 1) * T::kRow) = f2_unpack(acc.a.n);
                } else {
                    *reinterpret_cast<double2 *>(parts + u * T::kRow) = acc.store();
                }
            }
            __syncthreads();
            // 4. components in FP64: runs with their coefficients, the scaling
            // undone, phases, the tile's sites by a fixed xor tree
            double2 *partial = partial_base + B.partial_off[li];
            for (int c = warp; c < P.n_comp; c += kMinorWarps) {
                double re = 0.0, im = 0.0;
                for (int r = __ldg(P.run_off + c); r < __ldg(P.run_off + c + 1); ++r) {
                    double2 v;
                    if constexpr (kMx) {
                        MixedTraits::Acc a;
                        a.zero();
                        for (int u = r * per; u < (r + 1) * per; ++u) {
                            const float2 r0 = *reinterpret_cast<const float2 *>(parts + 2 * u * T::kRow);
                            const float2 r1 = *reinterpret_cast<const float2 *>(parts + (2 * u + 1) * T::kRow);
                            a.add(r0.x, r1.x, r0.y, r1.y);
                        }
                        v = a.value();
                    } else {
                        v = make_double2(0.0, 0.0);
                        for (int u = r * per; u < (r + 1) * per; ++u)
                            v = cadd(v, *reinterpret_cast<const double2 *>(parts + u * T::kRow));
                    }
                    const double coef = __ldg(P.run_coef + r);
                    re = __fma_rn(coef, v.x, re);
                    im = __fma_rn(coef, v.y, im);
                }
                const double inv_norm = __ldg(P.comp_inv_norm + c);
                re *= inv_norm;
                im *= inv_norm;
                if constexpr (kMx) {
                    const int ue = -__ldg(P.comp_deg + c) * se;
                    re = scalbn(re, ue);
                    im = scalbn(im, ue);
                }
                for (int q = 0; q < M.n_mom; ++q) {
                    const double2 ph = live ? site_phase(phase, site, M.n_mom, q) : make_double2(0, 0);
                    double pr = live ? __fma_rn(ph.x, re, -ph.y * im) : 0.0, pi = live ? __fma_rn(ph.x, im, ph.y * re) : 0.0;
                    for (int off = 16; off > 0; off >>= 1) {
                        pr += __shfl_xor_sync(0xffffffffu, pr, off);
                        pi += __shfl_xor_sync(0xffffffffu, pi, off);
                    }
                    if (lane == 0) partial[tile * (int64_t)(M.n_mom * P.n_comp) + q * P.n_comp + c] = make_double2(pr, pi);
                }
            }
            __syncthreads();  // the parts and minors are read before the next list or tile writes them
        }
    }
}

}  // namespace mbc
