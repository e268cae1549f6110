// Pair form of a nucleus with one or two baryons of each species (plan.h):
// C = sum_ij P_i Lambda_ij N_j with P and N the ordered products of a species'
// blocks, one sparse real Lambda per group of components.
//
//   k_pair      a warp takes a unit - a chunk of a group's Lambda rows for up to
//               MP proton and MN neutron spin sets - and a site group (32
//               sites; 64 in mixed precision, two per lane). Per row it sums
//               y_b = sum_j Lambda_ij N_b[j] over the row's entries, then adds
//               P_a[i] y_b to MP x MN accumulators. Site groups are the slow
//               index of the items, so the warps of the GPU gather from one
//               group's products at a time and those stay in L2.
//   k_pair_sum  adds the units' partial sums of every component in a fixed
//               order and undoes the mixed path's scaling.
// FP64 is bound by the FP64 pipe, mixed by the L2 gathers of N. Whole calls on
// GB300 against the recursion (8.5 M complex multiply-adds per site for one
// component, here 0.37 M for the products and 0.31 M real-complex ones; 531 M
// for all 1296): one component mixed, 16^3 x 4, 125.2 -> 12.1 ms; all, FP64, 64
// sites, 233.7 -> 26.9 ms; all, mixed, 512 sites, 227.7 -> 70.8 ms.
#pragma once

#include "large_kernel.cuh"

namespace mbc {

// One unit: rows [row0, row1) of Lambda (entries [e0, e1)), proton elements
// mp[0, na), neutron elements mn[0, nb); the partial of (a, b) goes to slot
// slot + a * stride_a + b * stride_b.
struct PairUnit {
    int64_t e0, e1;
    int32_t row0;
    int32_t na, nb;
    int32_t mp[6], mn[6];
    int32_t slot, stride_a, stride_b;
};

struct PairArgs {
    const PairUnit *units;
    int32_t n_units;
    const uint32_t *row_id;
    const uint32_t *col;   // N row, bit 31: last entry of its Lambda row
    const double *val;
    int64_t p_rows, n_rows;  // rows per element
};

struct __align__(16) PairRec {
    uint32_t col, last;
    double val;
};

// y += v x with a real factor, complex FP64
struct RealAcc64 {
    double re, im;
    __device__ __forceinline__ void zero() { re = im = 0.0; }
    __device__ __forceinline__ void add(double2 x, double v) {
        re = __fma_rn(v, x.x, re);
        im = __fma_rn(v, x.y, im);
    }
    __device__ __forceinline__ double2 store() const { return make_double2(re, im); }
};

template <int MP, int MN>
__global__ void __launch_bounds__(256) k_pair_fp64(PairArgs A, int W, const double2 *__restrict__ P,
                                                   const double2 *__restrict__ N, double2 *__restrict__ part) {
    __shared__ PairRec recs[8][32];
    const int lane = threadIdx.x & 31;
    PairRec *rec = recs[threadIdx.x >> 5];
    const int64_t n_items = (int64_t)A.n_units * (W >> 5);
    for (int64_t item = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5); item < n_items; item += (int64_t)gridDim.x * 8) {
        const PairUnit &u = A.units[item % A.n_units];
        const int col0 = (int)(item / A.n_units) * 32 + lane;
        const double2 *Nb[MN];
#pragma unroll
        for (int b = 0; b < MN; ++b) Nb[b] = N + (int64_t)u.mn[min(b, u.nb - 1)] * A.n_rows * W + col0;
        const double2 *Pb[MP];
#pragma unroll
        for (int a = 0; a < MP; ++a) Pb[a] = P + (int64_t)u.mp[min(a, u.na - 1)] * A.p_rows * W + col0;
        RealAcc64 y[MN];
        FP64Traits::Acc acc[MP][MN];
#pragma unroll
        for (int b = 0; b < MN; ++b) {
            y[b].zero();
#pragma unroll
            for (int a = 0; a < MP; ++a) acc[a][b].zero();
        }
        const uint32_t *row = A.row_id + u.row0;
        for (int64_t e0 = u.e0; e0 < u.e1; e0 += 32) {
            const int n = (int)min((int64_t)32, u.e1 - e0);
            __syncwarp();
            if (lane < n) {
                const uint32_t c = __ldg(A.col + e0 + lane);
                rec[lane] = PairRec{c & 0x7fffffffu, c >> 31, __ldg(A.val + e0 + lane)};
            }
            __syncwarp();
            constexpr int G = MN > 2 ? 1 : 4;
            for (int t = 0; t < n; t += G) {
                double2 x[G][MN];
#pragma unroll
                for (int g = 0; g < G; ++g)
                    if (t + g < n) {
                        const int64_t o = (int64_t)rec[t + g].col * W;
#pragma unroll
                        for (int b = 0; b < MN; ++b) x[g][b] = __ldg(Nb[b] + o);
                    }
#pragma unroll
                for (int g = 0; g < G; ++g) {
                    if (t + g >= n) break;
                    const PairRec r = rec[t + g];
#pragma unroll
                    for (int b = 0; b < MN; ++b) y[b].add(x[g][b], r.val);
                    if (r.last) {
                        const int64_t o = (int64_t)__ldg(row++) * W;
#pragma unroll
                        for (int a = 0; a < MP; ++a) {
                            const double2 p = __ldg(Pb[a] + o);
#pragma unroll
                            for (int b = 0; b < MN; ++b) acc[a][b].fma(p, y[b].store(), 0u);
                        }
#pragma unroll
                        for (int b = 0; b < MN; ++b) y[b].zero();
                    }
                }
            }
        }
#pragma unroll
        for (int a = 0; a < MP; ++a)
#pragma unroll
            for (int b = 0; b < MN; ++b)
                if (a < u.na && b < u.nb)
                    part[(int64_t)(u.slot + a * u.stride_a + b * u.stride_b) * W + col0] = acc[a][b].value();
    }
}

// The mixed form: two sites per lane, compensated FP32 sums (PairAcc). A row
// sum's terms enter the Kahan step as fma(x, v, n): one rounding each, as the
// signed step of PairAcc with a factor in the place of the sign.
struct RealAccPair {
    uint64_t sr, si, nr, ni;
    __device__ __forceinline__ void zero() { sr = si = nr = ni = 0ull; }
    __device__ __forceinline__ void add(ulonglong2 x, uint64_t v) {
        f2_kahan_signed(sr, nr, x.x, v);
        f2_kahan_signed(si, ni, x.y, v);
    }
    __device__ __forceinline__ ulonglong2 store() const { return make_ulonglong2(f2_add(sr, nr), f2_add(si, ni)); }
};

template <int MP, int MN>
__global__ void __launch_bounds__(128, MP * MN > 4 ? 3 : 6)
    k_pair_mx(PairArgs A, int W, const float2 *__restrict__ P, const float2 *__restrict__ N,
              double2 *__restrict__ part) {
    __shared__ OpRec recs[4][32];  // x: N row, y: last, sg: the value twice
    const int lane = threadIdx.x & 31;
    OpRec *rec = recs[threadIdx.x >> 5];
    const int64_t n_items = (int64_t)A.n_units * (W >> 6);
    const uint32_t row_bytes = (uint32_t)W * (uint32_t)sizeof(float2);
    for (int64_t item = (int64_t)blockIdx.x * 4 + (threadIdx.x >> 5); item < n_items; item += (int64_t)gridDim.x * 4) {
        const PairUnit &u = A.units[item % A.n_units];
        const int grp = (int)(item / A.n_units);
        const unsigned char *Nb[MN], *Pb[MP];
#pragma unroll
        for (int b = 0; b < MN; ++b)
            Nb[b] = reinterpret_cast<const unsigned char *>(N + (int64_t)u.mn[min(b, u.nb - 1)] * A.n_rows * W) +
                    grp * 512 + lane * 16;
#pragma unroll
        for (int a = 0; a < MP; ++a)
            Pb[a] = reinterpret_cast<const unsigned char *>(P + (int64_t)u.mp[min(a, u.na - 1)] * A.p_rows * W) +
                    grp * 512 + lane * 16;
        RealAccPair y[MN];
        PairAcc acc[MP][MN];
#pragma unroll
        for (int b = 0; b < MN; ++b) {
            y[b].zero();
#pragma unroll
            for (int a = 0; a < MP; ++a) acc[a][b].zero();
        }
        const uint64_t one = f2_sign_pair(false);
        const uint32_t *row = A.row_id + u.row0;
        for (int64_t e0 = u.e0; e0 < u.e1; e0 += 32) {
            const int n = (int)min((int64_t)32, u.e1 - e0);
            __syncwarp();
            if (lane < n) {
                const uint32_t c = __ldg(A.col + e0 + lane);
                const float v = (float)__ldg(A.val + e0 + lane);
                rec[lane] = OpRec{c & 0x7fffffffu, c >> 31, f2_pack(v, v)};
            }
            __syncwarp();
            constexpr int G = MN > 2 ? 2 : 8 / MN;
            for (int t = 0; t < n; t += G) {
                ulonglong2 x[G][MN];
#pragma unroll
                for (int g = 0; g < G; ++g)
                    if (t + g < n) {
                        const size_t o = (size_t)rec[t + g].x * row_bytes;
#pragma unroll
                        for (int b = 0; b < MN; ++b) x[g][b] = __ldg(reinterpret_cast<const ulonglong2 *>(Nb[b] + o));
                    }
#pragma unroll
                for (int g = 0; g < G; ++g) {
                    if (t + g >= n) break;
                    const OpRec r = rec[t + g];
#pragma unroll
                    for (int b = 0; b < MN; ++b) y[b].add(x[g][b], r.sg);
                    if (r.y) {
                        const size_t o = (size_t)__ldg(row++) * row_bytes;
#pragma unroll
                        for (int a = 0; a < MP; ++a) {
                            const ulonglong2 p = __ldg(reinterpret_cast<const ulonglong2 *>(Pb[a] + o));
#pragma unroll
                            for (int b = 0; b < MN; ++b) acc[a][b].fma(p, y[b].store(), one);
                        }
#pragma unroll
                        for (int b = 0; b < MN; ++b) y[b].zero();
                    }
                }
            }
        }
        const int col0 = grp * 64 + 2 * lane;
#pragma unroll
        for (int a = 0; a < MP; ++a)
#pragma unroll
            for (int b = 0; b < MN; ++b)
                if (a < u.na && b < u.nb) {
                    double2 *dst = part + (int64_t)(u.slot + a * u.stride_a + b * u.stride_b) * W + col0;
                    const float2 sr = f2_unpack(acc[a][b].sr), si = f2_unpack(acc[a][b].si);
                    const float2 nr = f2_unpack(acc[a][b].nr), ni = f2_unpack(acc[a][b].ni);
                    dst[0] = make_double2((double)sr.x + (double)nr.x, (double)si.x + (double)ni.x);
                    dst[1] = make_double2((double)sr.y + (double)nr.y, (double)si.y + (double)ni.y);
                }
    }
}

// Cout[comp][site]: the partials of the component's evaluations (slots
// [slot_off[ev], slot_off[ev + 1])), warp w of the CTA adding slots w, w + 32,
// ..., the warps' sums then in warp order. FP64: an SM's four FP64 units take a
// warp's addition 64 cycles each, hence 32 warps per 32 sites.
__global__ void __launch_bounds__(1024) k_pair_sum(const int32_t *__restrict__ comp_off,
                                                   const int32_t *__restrict__ comp_eval,
                                                   const int32_t *__restrict__ slot_off, int W,
                                                   const double2 *__restrict__ part, const int32_t *__restrict__ sexp,
                                                   int degree, double scale, double2 *__restrict__ Cout) {
    __shared__ double2 sums[32][33];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, c = blockIdx.x;
    const int col = blockIdx.y * 32 + lane;
    double2 s = make_double2(0.0, 0.0);
    for (int k = comp_off[c]; k < comp_off[c + 1]; ++k) {
        const int ev = comp_eval[k];
        for (int t = slot_off[ev] + warp; t < slot_off[ev + 1]; t += 32) s = cadd(s, part[(int64_t)t * W + col]);
    }
    sums[warp][lane] = s;
    __syncthreads();
    // transposed: warp w adds the 32 sums of site w by a fixed tree
    s = sums[lane][warp];
    for (int off = 16; off > 0; off >>= 1) {
        s.x += __shfl_xor_sync(0xffffffffu, s.x, off);
        s.y += __shfl_xor_sync(0xffffffffu, s.y, off);
    }
    if (lane == 0) {
        const int site = blockIdx.y * 32 + warp, ue = -degree * sexp[site];
        Cout[(int64_t)c * W + site] = make_double2(scalbn(s.x * scale, ue), scalbn(s.y * scale, ue));
    }
}

}  // namespace mbc
