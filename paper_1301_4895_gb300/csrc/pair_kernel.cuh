// Pair form of a nucleus with one or two baryons of each species (plan.h):
// C = sum_ij P_i Lambda_ij N_j with P and N the ordered products of a species'
// blocks, one sparse real Lambda per group of components.
//
// Blocks and products lie in tiles of a warp's sites, [tile][row][32 sites of
// FP64 or 64 of FP32], 512 B a row.
//   k_pair_prod a CTA copies the 4 x n_pairs block rows that the products with
//               two given singles name into shared memory (135 KB) and forms the
//               range's products from there; from L2 their operands would need
//               its whole bandwidth in mixed precision.
//   k_pair      a CTA takes a unit - packs of rows of one group for up to MR spin
//               sets of the row side and MG of the gathered side (a P row
//               gathers N, an N row gathers P) - and a tile. A pack is rows that
//               name at most kPackCols distinct gathered entries; the CTA copies
//               those into shared memory, then a warp takes a row at a time: y_b
//               = sum_j Lambda_ij G_b[j] from shared memory, then R_a[i] y_b into
//               MR x MG accumulators, R_a[i] loaded while y is summed. Gathering
//               from L2 instead left the warps waiting (11 cycles an
//               instruction, L1 hits 57 %).
//   k_pair_sum  adds the units' partial sums of every component in a fixed
//               order and undoes the mixed path's scaling.
// Mixed sums are compensated FP32 throughout, the contraction's too, which the
// recursion makes in FP64. Median errors against FP64 at single sites (eps = 0.05),
// against the recursion on FP32 blocks: 9.4e-8 -> 6.9e-8 (one component), 1.44e-7 ->
// 9.5e-8 (all); the blocks, from exact products, round once.
// FP64 is bound by the FP64 pipe, mixed by shared-memory wavefronts (53-66 % of
// the pipe) and its few warps' latencies. Whole calls on GB300 against the
// recursion (8.5 M complex multiply-adds per site for one component, here 0.37 M
// for the products and 0.31 M real-complex ones; 531 M for all 1296): one
// component mixed, 16^3 x 4, 125.2 -> 7.9 ms; all, FP64, 64 sites, 233.7 -> 19.5
// ms; all, mixed, 512 sites, 210.1 -> 19.9 ms. With L2 gathers and rows in rank
// order 12.1, 26.9 and 70.8; with rows staged through registers (one load's
// latency per row and warp, 10 % of a pack's time) 9.35, 20.0 and 24.2.
#pragma once

#include "large_kernel.cuh"
#include "plan.h"

namespace mbc {

constexpr int kTile64 = 32, kTileMx = 64;  // sites per tile
// warps per CTA of k_pair_prod: what its registers allow
template <bool MX>
constexpr int kProdWarps = MX ? 16 : 24;

// Products of one (tile, spin set, singles range) per CTA; grid = tiles x sets x
// ranges. A warp takes runs of rows that share a quark triple: the triple's pairs
// (12 of a row's 24 operands) stay in registers, and a row's other pairs are at
// fixed distances from three addresses. With 24 operands read and 24 addresses
// decoded for each row the mixed kernel was held by issue and the shared-memory
// pipe: 3.68 -> 2.97 ms of a one-component 4He call on 16^3 x 4 sites (3.06 with 20
// warps and the negated imaginary parts formed per term). FP64 is bound by its pipe
// either way.
template <bool MX, int NPAIR>
__global__ void __launch_bounds__(32 * kProdWarps<MX>, 1)
    k_pair_prod(const uint2 *__restrict__ runs, const int32_t *__restrict__ run_off, const uint32_t *__restrict__ recs,
                const int32_t *__restrict__ range_off, const uint16_t *__restrict__ range_e, int n_ranges,
                const uint32_t *__restrict__ masks, int n_masks, int nxi, int64_t block_rows, int n_rows,
                const ulonglong2 *__restrict__ f, ulonglong2 *__restrict__ prod) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    using V = std::conditional_t<MX, ulonglong2, double2>;
    ulonglong2 *rows = reinterpret_cast<ulonglong2 *>(smem_raw);  // [f | g][single][pair][lane]
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int k = blockIdx.x % n_ranges, m = blockIdx.x / n_ranges % n_masks;
    const int64_t tile = blockIdx.x / n_ranges / n_masks;
    const uint32_t mask = __ldg(masks + m);
    const int s0 = __ffs(mask) - 1, s1 = 31 - __clz(mask), e0 = range_e[k] & 255, e1 = range_e[k] >> 8;
    const ulonglong2 *ft = f + tile * block_rows * 32;
    for (int r = warp; r < 4 * NPAIR; r += kProdWarps<MX>) {
        const int s = r / (2 * NPAIR), i = r / NPAIR & 1, p = r % NPAIR;
        async_copy16(rows + r * 32 + lane, ft + ((int64_t)((s ? s1 : s0) * NPAIR + p) * nxi + (i ? e1 : e0)) * 32 + lane);
    }
    async_copy_wait_all();
    __syncthreads();
    const V *R = reinterpret_cast<const V *>(rows) + lane;
    // f (s = 0) or g (s = 1) with single i
    auto at = [](const V *pair, int s, int i) { return pair[(2 * s + i) * NPAIR * 32]; };
    ulonglong2 *out = prod + ((tile * n_masks + m) * n_rows + range_off[k]) * 32 + lane;
    // a run goes to one warp; in FP64 row by row, since its pipe wants equal warps
    // and not fewer operands (5.07 against 5.11 ms in a batch on 24^3 sites)
    constexpr int kPart = MX ? PairPlan::kProdRun : 1;
    const int n_runs = run_off[k + 1] - run_off[k];
    runs += run_off[k];
    for (int u = warp; u < n_runs * ((PairPlan::kProdRun + kPart - 1) / kPart); u += kProdWarps<MX>) {
        const uint2 run = __ldg(runs + u % n_runs);
        const int t0 = u / n_runs * kPart, n = min((int)(run.y & 255u), t0 + kPart);
        if (t0 >= n) continue;
        const uint32_t mine = lane < n ? __ldg(recs + run.x + lane) : 0u;
        V held[3][2][2];
#pragma unroll
        for (int q = 0; q < 3; ++q)
#pragma unroll
            for (int s = 0; s < 2; ++s)
#pragma unroll
                for (int i = 0; i < 2; ++i) held[q][s][i] = at(R + (run.y >> (8 * q + 8) & 255u) * 32, s, i);
        uint64_t neg_im[MX ? 3 : 1][2][2];  // -Im held
        if constexpr (MX) {
#pragma unroll
            for (int q = 0; q < 3; ++q)
#pragma unroll
                for (int s = 0; s < 2; ++s)
#pragma unroll
                    for (int i = 0; i < 2; ++i) neg_im[q][s][i] = f2_neg(held[q][s][i].y);
        }
        for (int t = t0; t < n; ++t) {
            const uint32_t rec = __shfl_sync(0xffffffffu, mine, t), odd = rec >> 30;
            ulonglong2 *to = out + (int64_t)(rec >> 21 & 511u) * 32;
            std::conditional_t<MX, PairAcc, FP64Traits::Acc> acc;
            acc.zero();
#pragma unroll
            for (int q = 0; q < 3; ++q) {
                const V *pair = R + (rec >> (7 * q) & 127u) * 32;
#pragma unroll
                for (int i = 0; i < 2; ++i) {  // f takes single i, g the other: e1 | e0 is odd
                    const bool neg = (odd == (uint32_t)q) != (i == 1);
                    if constexpr (MX) {
                        const uint64_t sg = f2_sign_pair(neg);
                        acc.fma(at(pair, 1, 1 - i), held[q][0][i], neg_im[q][0][i], sg);
                        acc.fma(at(pair, 0, i), held[q][1][1 - i], neg_im[q][1][1 - i], sg);
                    } else {
                        const uint32_t sg = neg ? 0x80000000u : 0u;
                        acc.fma(held[q][0][i], at(pair, 1, 1 - i), sg);
                        acc.fma(at(pair, 0, i), held[q][1][1 - i], sg);
                    }
                }
            }
            *reinterpret_cast<V *>(to) = acc.store();
        }
    }
}

struct PairPack {
    int64_t row0;    // rows [row0, row0 + n_rows)
    int64_t col0;    // gathered rows cols[col0 .. col0 + n_cols)
    int32_t n_rows, n_cols;
};
// One unit: packs [pack0, pack1), row-side elements re[0, nr), gathered
// elements ge[0, ng) (swap: rows of N gathering P); the partial of (a, b) goes
// to slot + a * stride_r + b * stride_g.
struct PairUnit {
    int32_t pack0, pack1, swap;
    int32_t nr, ng;
    int32_t re[6], ge[6];
    int32_t slot, stride_r, stride_g;
};
struct __align__(8) PairRow {
    uint32_t row_n;  // row-side row | entries << 24
    uint32_t e0;     // first entry
    __host__ __device__ uint32_t row() const { return row_n & 0xffffffu; }
    __host__ __device__ uint32_t n() const { return row_n >> 24; }
};
static_assert(kPackCols < 256, "PairRow::n");

struct PairArgs {
    const PairUnit *units;
    int32_t n_units, n_tiles;
    const PairPack *packs;
    const PairRow *rows;
    const uint32_t *cols;
    const uint16_t *slot;      // entries: position of the gathered row in its pack
    const double *val;
    int64_t p_rows, n_rows;    // rows per element
    int64_t p_tile, n_tile;    // rows per tile of P's and N's buffer
};

// y += v x with a real factor v, and acc += x y; values of 16 B per lane: one
// site in FP64, two in mixed precision. Mixed terms of y enter the Kahan step as
// fma(x, v, n): one rounding each, as PairAcc's signed step with a factor in the
// place of the sign.
struct Pair64 {
    static constexpr int kSites = 1;
    struct Y {
        double re, im;
        __device__ __forceinline__ void zero() { re = im = 0.0; }
        __device__ __forceinline__ void add(ulonglong2 x, double v) {
            re = __fma_rn(v, __longlong_as_double((long long)x.x), re);
            im = __fma_rn(v, __longlong_as_double((long long)x.y), im);
        }
    };
    struct Acc {
        FP64Traits::Acc a;
        __device__ __forceinline__ void zero() { a.zero(); }
        __device__ __forceinline__ void fma(ulonglong2 x, const Y &y) {
            a.fma(make_double2(__longlong_as_double((long long)x.x), __longlong_as_double((long long)x.y)),
                  make_double2(y.re, y.im), 0u);
        }
        __device__ __forceinline__ void values(double2 (&v)[1]) const { v[0] = a.value(); }
    };
    // record of an entry: place of the gathered row, value
    struct __align__(16) Rec {
        uint32_t off, pad;
        double v;
    };
    __device__ __forceinline__ static Rec rec(uint32_t off, double v) { return Rec{off, 0u, v}; }
    static constexpr int kRead = 1;  // records per load
    __device__ __forceinline__ static void read(const Rec *r, uint32_t (&off)[1], double (&v)[1]) {
        const Rec w = *r;
        off[0] = w.off;
        v[0] = w.v;
    }
    using Factor = double;
};
struct PairMx {
    static constexpr int kSites = 2;
    struct Y {
        uint64_t sr, si, nr, ni;
        __device__ __forceinline__ void zero() { sr = si = nr = ni = 0ull; }
        __device__ __forceinline__ void add(ulonglong2 x, uint64_t v) {
            f2_kahan_signed(sr, nr, x.x, v);
            f2_kahan_signed(si, ni, x.y, v);
        }
    };
    struct Acc {
        PairAcc a;
        __device__ __forceinline__ void zero() { a.zero(); }
        __device__ __forceinline__ void fma(ulonglong2 x, const Y &y) {
            a.fma(x, make_ulonglong2(f2_add(y.sr, y.nr), f2_add(y.si, y.ni)), f2_sign_pair(false));
        }
        __device__ __forceinline__ void values(double2 (&v)[2]) const {
            const float2 sr = f2_unpack(a.sr), si = f2_unpack(a.si), nr = f2_unpack(a.nr), ni = f2_unpack(a.ni);
            v[0] = make_double2((double)sr.x + (double)nr.x, (double)si.x + (double)ni.x);
            v[1] = make_double2((double)sr.y + (double)nr.y, (double)si.y + (double)ni.y);
        }
    };
    using Rec = uint2;  // 8 B, two in one broadcast load
    static constexpr int kRead = 2;
    __device__ __forceinline__ static Rec rec(uint32_t off, double v) { return make_uint2(off, __float_as_uint((float)v)); }
    __device__ __forceinline__ static void read(const Rec *r, uint32_t (&off)[2], uint64_t (&v)[2]) {
        const uint4 w = *reinterpret_cast<const uint4 *>(r);
        off[0] = w.x;
        v[0] = f2_pack(__uint_as_float(w.y), __uint_as_float(w.y));
        off[1] = w.z;
        v[1] = f2_pack(__uint_as_float(w.w), __uint_as_float(w.w));
    }
    using Factor = uint64_t;
};

// Row-side values a warp holds in registers while it sums y; the others of MR
// (six spin sets, mixed: the accumulators leave no room) come by its own copies
// through shared memory meanwhile (all components, mixed, 512 sites: 19.0 ms, 19.3
// where they are loaded after y).
template <class T, int MR>
__host__ __device__ constexpr int pair_held() {
    return T::kSites == 1 || MR <= 2 ? MR : MR / 2;
}
// dynamic shared memory: the pack's rows [MG][kPackCols][32 lanes], 32 records per
// warp, its row-side values [MR - held][32 lanes]; the partial sums of a unit reuse
// the pack's room
template <class T, int MR, int MG, int WARPS>
__host__ __device__ constexpr size_t pair_smem() {
    return (size_t)MG * kPackCols * 512 +
           (size_t)WARPS * (32 * sizeof(typename T::Rec) + (MR - pair_held<T, MR>()) * 512);
}

template <class T, int MR, int MG, int WARPS>
__global__ void __launch_bounds__(32 * WARPS, MG == 1 ? 2 : 1)
    k_pair(PairArgs A, int W, const ulonglong2 *__restrict__ P, const ulonglong2 *__restrict__ N,
           double2 *__restrict__ part) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    ulonglong2 *stage = reinterpret_cast<ulonglong2 *>(smem_raw);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    typename T::Rec *rec = reinterpret_cast<typename T::Rec *>(smem_raw + (size_t)MG * kPackCols * 512) + warp * 32;
    ulonglong2 *xs = reinterpret_cast<ulonglong2 *>(smem_raw + (size_t)MG * kPackCols * 512 +
                                                    (size_t)WARPS * 32 * sizeof(typename T::Rec)) +
                     warp * (MR - pair_held<T, MR>()) * 32 + lane;
    __shared__ uint32_t Ro[MR];
    const int64_t n_items = (int64_t)A.n_units * A.n_tiles;
    for (int64_t item = blockIdx.x; item < n_items; item += gridDim.x) {
        const PairUnit &u = A.units[item % A.n_units];
        const int64_t tile = item / A.n_units;
        const ulonglong2 *Pt = P + tile * A.p_tile * 32 + lane, *Nt = N + tile * A.n_tile * 32 + lane;
        const ulonglong2 *Rs = u.swap ? Nt : Pt, *Gs = u.swap ? Pt : Nt;
        const int64_t r_rows = u.swap ? A.n_rows : A.p_rows, g_rows = u.swap ? A.p_rows : A.n_rows;
        // 16-byte words from Rs (shared memory: registers are short in the mixed form)
        if (threadIdx.x < MR) Ro[threadIdx.x] = (uint32_t)(u.re[min((int)threadIdx.x, u.nr - 1)] * r_rows) * 32u;
        constexpr int H = pair_held<T, MR>();
        typename T::Acc acc[MR][MG];
#pragma unroll
        for (int a = 0; a < MR; ++a)
#pragma unroll
            for (int b = 0; b < MG; ++b) acc[a][b].zero();
        for (int k = u.pack0; k < u.pack1; ++k) {
            const PairPack pk = A.packs[k];
            __syncthreads();  // the previous pack (or unit) is done with the rows
            static_assert(kPackCols <= 32 * WARPS, "a lane holds one of its warp's columns");
            const uint32_t mine = warp + WARPS * lane < pk.n_cols ? __ldg(A.cols + pk.col0 + warp + WARPS * lane) : 0u;
            for (int c = warp, i = 0; c < pk.n_cols; c += WARPS, ++i) {
                const int64_t row = (int64_t)__shfl_sync(0xffffffffu, mine, i) * 32;
#pragma unroll
                for (int b = 0; b < MG; ++b)
                    async_copy16(stage + (b * kPackCols + c) * 32 + lane,
                                 Gs + (int64_t)u.ge[min(b, u.ng - 1)] * g_rows * 32 + row);
            }
            async_copy_wait_all();
            __syncthreads();
            const ulonglong2 *G = stage + lane;
            // two rows ahead: the next row's records are loaded while this one is
            // worked off, and the row after gives their place
            const PairRow none{0u, 0u};
            const PairRow *rows = A.rows + pk.row0;
            PairRow row = warp < pk.n_rows ? rows[warp] : none;
            PairRow next = warp + WARPS < pk.n_rows ? rows[warp + WARPS] : none;
            auto load = [&](const PairRow &w, uint32_t e0, double &v, uint32_t &o) {
                if (e0 + lane < w.n()) {
                    v = __ldg(A.val + w.e0 + e0 + lane);
                    o = __ldg(A.slot + w.e0 + e0 + lane);
                }
            };
            double rv = 0.0;
            uint32_t ro = 0;
            load(row, 0, rv, ro);
            for (int r = warp; r < pk.n_rows; r += WARPS) {
                const ulonglong2 *Rr = Rs + row.row() * 32u;
                ulonglong2 x[H];
#pragma unroll
                for (int a = 0; a < H; ++a) x[a] = __ldg(Rr + Ro[a]);
#pragma unroll
                for (int a = H; a < MR; ++a) async_copy16(xs + (a - H) * 32, Rr + Ro[a]);
                const PairRow after = r + 2 * WARPS < pk.n_rows ? rows[r + 2 * WARPS] : none;
                typename T::Y y[MG];
#pragma unroll
                for (int b = 0; b < MG; ++b) y[b].zero();
                for (uint32_t e0 = 0; e0 < row.n(); e0 += 32) {
                    const int n = (int)min(32u, row.n() - e0);
                    __syncwarp();
                    rec[lane] = T::rec(ro * 32u, rv);
                    __syncwarp();
                    if (e0 + 32 < row.n())
                        load(row, e0 + 32, rv, ro);
                    else
                        load(next, 0, rv, ro);
                    constexpr int K = T::kRead;
                    int t = 0;
                    for (; t + 4 <= n; t += 4) {
#pragma unroll
                        for (int g = 0; g < 4; g += K) {
                            uint32_t off[K];
                            typename T::Factor v[K];
                            T::read(rec + t + g, off, v);
#pragma unroll
                            for (int q = 0; q < K; ++q)
#pragma unroll
                                for (int b = 0; b < MG; ++b) y[b].add(G[b * kPackCols * 32 + off[q]], v[q]);
                        }
                    }
                    for (; t < n; t += K) {  // a record beyond n is not used
                        uint32_t off[K];
                        typename T::Factor v[K];
                        T::read(rec + t, off, v);
#pragma unroll
                        for (int q = 0; q < K; ++q)
                            if (t + q < n)
#pragma unroll
                                for (int b = 0; b < MG; ++b) y[b].add(G[b * kPackCols * 32 + off[q]], v[q]);
                    }
                }
#pragma unroll
                for (int a = 0; a < H; ++a)
#pragma unroll
                    for (int b = 0; b < MG; ++b) acc[a][b].fma(x[a], y[b]);
                if constexpr (H < MR) async_copy_wait_all();  // a lane reads what it copied
#pragma unroll
                for (int a = H; a < MR; ++a) {
                    const ulonglong2 v = xs[(a - H) * 32];
#pragma unroll
                    for (int b = 0; b < MG; ++b) acc[a][b].fma(v, y[b]);
                }
                row = next;
                next = after;
            }
        }
        // the unit's partial: the warps' sums added in warp order, a pair (a, b)
        // per round of MG
        constexpr int S = T::kSites;
        double2 *sums = reinterpret_cast<double2 *>(smem_raw);  // [MG][WARPS][32 S]
#pragma unroll
        for (int a = 0; a < MR; ++a) {
            __syncthreads();
#pragma unroll
            for (int b = 0; b < MG; ++b) {
                double2 v[S];
                acc[a][b].values(v);
#pragma unroll
                for (int q = 0; q < S; ++q) sums[(b * WARPS + warp) * 32 * S + lane * S + q] = v[q];
            }
            __syncthreads();
            for (int o = threadIdx.x; o < MG * 32 * S; o += 32 * WARPS) {
                const int b = o / (32 * S), site = o % (32 * S);
                if (a >= u.nr || b >= u.ng) continue;
                double2 t = sums[b * WARPS * 32 * S + site];
                for (int w = 1; w < WARPS; ++w) t = cadd(t, sums[(b * WARPS + w) * 32 * S + site]);
                part[(int64_t)(u.slot + a * u.stride_r + b * u.stride_g) * W + tile * 32 * S + site] = t;
            }
        }
    }
}

// Cout[comp][site]: the partials of the component's evaluations (slots
// [slot_off[ev], slot_off[ev + 1])) of S sites per CTA: group g of G adds slots g,
// g + G, ..., the groups' sums then in a fixed order. An SM's four FP64 units take
// a warp's addition 64 cycles each, so the shape follows the work. Enough CTAs
// (all components): 32 sites, 4 groups, no tree - 0.09 ms for 512 sites, where 32
// warps and a tree per CTA took 0.91. Else (one component): 8 sites and 128 groups,
// which spreads the additions over the SMs - 6.2 us for 1,024 sites (10 with 4
// groups, 12.5 with 32 warps on 32 sites).
template <int S, int G>
__global__ void __launch_bounds__(S * G) k_pair_sum(const int32_t *__restrict__ comp_off,
                                                    const int32_t *__restrict__ comp_eval,
                                                    const int32_t *__restrict__ slot_off, int W,
                                                    const double2 *__restrict__ part, const int32_t *__restrict__ sexp,
                                                    int degree, double scale, double2 *__restrict__ Cout) {
    __shared__ double2 sums[G][S + 1];
    const int site = threadIdx.x % S, g = threadIdx.x / S, c = blockIdx.x;
    const int col = blockIdx.y * S + site;
    double2 s = make_double2(0.0, 0.0);
    for (int k = comp_off[c]; k < comp_off[c + 1]; ++k) {
        const int ev = comp_eval[k];
        for (int t = slot_off[ev] + g; t < slot_off[ev + 1]; t += G) s = cadd(s, part[(int64_t)t * W + col]);
    }
    sums[g][site] = s;
    __syncthreads();
    int out = -1;  // the site this thread writes
    if constexpr (G <= 8) {
        if (g == 0) {
            for (int q = 1; q < G; ++q) s = cadd(s, sums[q][site]);
            out = site;
        }
    } else {  // a warp per site: lane l adds groups l, l + 32, ..., then a fixed tree
        const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
        if (w < S) {
            s = sums[lane][w];
            for (int q = lane + 32; q < G; q += 32) s = cadd(s, sums[q][w]);
            for (int off = 16; off > 0; off >>= 1) {
                s.x += __shfl_xor_sync(0xffffffffu, s.x, off);
                s.y += __shfl_xor_sync(0xffffffffu, s.y, off);
            }
            if (lane == 0) out = w;
        }
    }
    if (out >= 0) {
        const int at = blockIdx.y * S + out, ue = -degree * sexp[at];
        Cout[(int64_t)c * W + at] = make_double2(scalbn(s.x * scale, ue), scalbn(s.y * scale, ue));
    }
}

}  // namespace mbc
