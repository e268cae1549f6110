// Momentum-projected blocks (Sec. 2: blocks carry a sink function s(x); here
// every baryon uses s(x) = exp(-2 pi i n.x / L)), then one recursion per
// (configuration, time slice, momentum) on the summed blocks.
//
// The block is f[alpha; i j; s] = g[alpha, i; j s] - g[alpha, j; i s] with
// g[alpha, i; j s] = sum_c S[alpha c, i] Q[c][j, s] and Q symmetric, so the site
// sums are taken over g (48 x 78 entries of 3 multiply-adds each, against 6 for
// each of f's 3168) and antisymmetrised once. Momentum phases factorise over a
// lattice line: sum_x e^{-2 pi i n_x x / L_x} g first, one sum per distinct n_x
// (plain additions for n_x = 0), then the line's phase per momentum.
//
//   k_line_phases   tables of the x phases and of the lines' phases;
//   k_project       a CTA walks a chunk of a slab's sites with the sums of 2 spins
//                   x 12 x 78 entries of g: the line's in registers (a thread: one
//                   (j, s), two i, both spins), the momenta's (up to 4) in shared
//                   memory, where the tiles and diquarks of a batch of sites pass
//                   too. 15 warps. Only chunk sums are written, where 16-site
//                   tiles wrote 0.2-0.4 GB;
//   k_project_sum   adds the chunks in order and antisymmetrises: f per (slab,
//                   momentum), and in mixed precision the largest entry per item;
//   k_load_proj_blocks copies the summed blocks of a wave of items into the
//                   layout of the wave kernels (MIXED: exact power-of-two scaling
//                   per item);
//   k_write_items   writes each item's contracted components to out.
// FP64 throughout in the FP64 path (bound by its pipe). The mixed path takes FP32
// products and compensated FP32 sums along a line; a line's sum enters the momenta
// in both words, with exact products and the line's phase in two words: rounded to one
// word before and after that product, a line of near-identity sites cost up to a third
// of the accuracy at momenta across the lines (median error of 4He rel at (0, 1, 0),
// eps = 0.05: 16^3 9.1e-7 -> 6.4e-7, 5 x 7 x 9 1.6e-6 -> 6.8e-7; blocks weighted by one
// FP32 phase per site 6.9e-7 and 1.4e-6; along the lines 7.6e-7 and 6.7e-7, an entry of
// g being rounded for two of f). 4 momenta on 16^3 x 4: 623 -> 633 us; lines whose
// phases are all ones only add (two sources on 16^3 x 16: 526 us as before, else 537).
#pragma once

#include "large_kernel.cuh"

namespace mbc {

constexpr int kProjMoms = 4;  // momenta per pass

// One pass of k_project: momenta q0 .. q0 + n_mom, their n_x among n_x distinct
// values; x phases in column xcol[k] of the x table (trivial: all ones). flat: the
// lines' phases of a momentum are all ones.
struct ProjPass {
    int32_t q0, n_mom, n_x;
    int32_t nx_of[kProjMoms], flat[kProjMoms], xcol[kProjMoms], trivial[kProjMoms];
};

// A phase table's entry in the mixed path: two FP32 words of a complex number.
struct Phase32 {
    float2 h, l;
};
static_assert(sizeof(Phase32) == sizeof(double2), "one table for both");

// xtab[x][d] = e^{-2 pi i D.mom[d][0] x / Lx}; ytab[y + Ly z][q] = the (y, z) phase
// of momentum q. Column d of xtab belongs to the d-th distinct n_x. words: entries as
// Phase32.
__global__ void k_line_phases(FieldDesc F, MomDesc M, MomDesc D, int words, double2 *xtab, double2 *ytab) {
    auto put = [&](double2 *to, double2 v) {
        if (words) {
            const float2 h = make_float2((float)v.x, (float)v.y);
            *reinterpret_cast<Phase32 *>(to) = Phase32{h, make_float2((float)(v.x - h.x), (float)(v.y - h.y))};
        } else {
            *to = v;
        }
    };
    const int nl = F.ly * F.lz;
    const int64_t total = (int64_t)F.lx * D.n_mom + (int64_t)nl * M.n_mom;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x) {
        if (i < (int64_t)F.lx * D.n_mom) {
            const int n[3] = {D.mom[i % D.n_mom][0], 0, 0};
            put(xtab + i, mom_phase(n, (int)(i / D.n_mom), 0, 0, F.lx, F.ly, F.lz));
        } else {
            const int64_t k = i - (int64_t)F.lx * D.n_mom;
            const int q = (int)(k % M.n_mom), line = (int)(k / M.n_mom);
            const int n[3] = {0, M.mom[q][1], M.mom[q][2]};
            put(ytab + k, mom_phase(n, 0, line % F.ly, line / F.ly, F.lx, F.ly, F.lz));
        }
    }
}

// Sums over a line's sites (acc += x, or ph x) and, Total, over the lines (acc += ph
// times a line's sum). Phase: a phase table's entry, first() what a site multiplies by.
struct ProjSum64 {
    using V = double2;
    using Phase = double2;
    double re, im;
    __device__ __forceinline__ static V first(Phase p) { return p; }
    __device__ __forceinline__ void zero() { re = im = 0.0; }
    __device__ __forceinline__ void add(V x) {
        re += x.x;
        im += x.y;
    }
    __device__ __forceinline__ void add(V ph, V x) {
        re = __fma_rn(ph.x, x.x, __fma_rn(-ph.y, x.y, re));
        im = __fma_rn(ph.x, x.y, __fma_rn(ph.y, x.x, im));
    }
    struct Total;
};
struct ProjSum64::Total {
    ProjSum64 s;
    __device__ __forceinline__ void zero() { s.zero(); }
    __device__ __forceinline__ void add(Phase ph, bool, const ProjSum64 &line) { s.add(ph, make_double2(line.re, line.im)); }
    __device__ __forceinline__ double2 value() const { return make_double2(s.re, s.im); }
};
struct ProjSumMx {
    using V = float2;
    using Phase = Phase32;
    MixedTraits::Acc a;
    __device__ __forceinline__ static V first(Phase p) { return p.h; }
    __device__ __forceinline__ void zero() { a.zero(); }
    __device__ __forceinline__ void add(V x) { f2_kahan(a.s, a.n, f2_pack(x.x, x.y)); }
    __device__ __forceinline__ void add(V ph, V x) { a.add_prod(ph, x); }
    struct Total {
        BlockAccMx b;
        __device__ __forceinline__ void zero() { b.zero(); }
        __device__ __forceinline__ void add(Phase ph, bool flat, const ProjSumMx &line) {
            const DiquarkMx y{f2_unpack(line.a.s), f2_unpack(line.a.n)};
            if (flat) {
                float2 e;
                two_sum(b.h.x, y.h.x, b.h.x, e.x);
                two_sum(b.h.y, y.h.y, b.h.y, e.y);
                b.l = make_float2(__fadd_rn(b.l.x, __fadd_rn(e.x, y.l.x)), __fadd_rn(b.l.y, __fadd_rn(e.y, y.l.y)));
                return;
            }
            b.add(ph.h, y);
            b.l.x = __fmaf_rn(ph.l.x, y.h.x, __fmaf_rn(-ph.l.y, y.h.y, b.l.x));
            b.l.y = __fmaf_rn(ph.l.x, y.h.y, __fmaf_rn(ph.l.y, y.h.x, b.l.y));
        }
        __device__ __forceinline__ double2 value() const {
            return make_double2((double)b.h.x + (double)b.l.x, (double)b.h.y + (double)b.l.y);
        }
    };
};

// (j, s) pairs, i values per thread, threads of one way (a walk over one chunk)
// and ways of a CTA (six walks share a CTA for 6 columns).
__host__ __device__ constexpr int proj_njs(int nxi) { return nxi * (nxi + 1) / 2; }
__host__ __device__ constexpr int proj_ipt(int nxi) { return nxi == 12 ? 2 : 3; }
__host__ __device__ constexpr int proj_way(int nxi) { return nxi / proj_ipt(nxi) * proj_njs(nxi); }
__host__ __device__ constexpr int proj_ways(int nxi) { return nxi == 12 ? 1 : 6; }
__host__ __device__ constexpr int proj_threads(int nxi) { return (proj_way(nxi) * proj_ways(nxi) + 31) / 32 * 32; }
// sites in shared memory at a time (a multiple of 2: 16-byte rows)
__host__ __device__ constexpr int proj_batch(bool mixed) { return mixed ? 8 : 4; }

inline size_t project_smem_bytes(int nrow, int nxi, int n_mom, bool mixed) {
    return (size_t)2 * proj_ipt(nxi) * n_mom * proj_threads(nxi) * 16 +
           (size_t)proj_ways(nxi) * proj_batch(mixed) * (nrow * nxi + 3 * proj_njs(nxi) + kProjMoms) * (mixed ? 8 : 16);
}

template <class Sum, int NXI, int NX>
__global__ void __launch_bounds__(proj_threads(NXI), 1)
    k_project(FieldDesc F, const __grid_constant__ ProjPass ps, const double2 *__restrict__ xtab, int n_dx,
              const double2 *__restrict__ ytab, int n_mom, int nrow, int n_g2, int n_chunks, int64_t n_ways,
              double2 *__restrict__ partial) {
    using V = typename Sum::V;
    using R = decltype(V::x);
    constexpr int NJS = proj_njs(NXI), WAY = proj_way(NXI), WAYS = proj_ways(NXI);
    constexpr int B = proj_batch(sizeof(V) == 8);
    constexpr int I = proj_ipt(NXI), O = 2 * I;  // outputs of a thread: (spin, i)
    constexpr int kProjThreads = proj_threads(NXI);
    using Total = typename Sum::Total;
    using Phase = typename Sum::Phase;
    static_assert(sizeof(Total) == 16, "sums in shared memory");
    extern __shared__ __align__(16) unsigned char smem_raw[];
    Total *out = reinterpret_cast<Total *>(smem_raw) + threadIdx.x;  // [mom][O][thread]
    const int nent = nrow * NXI, per_way = B * (nent + 3 * NJS + kProjMoms);
    const int wy = threadIdx.x / WAY, tw = threadIdx.x % WAY;
    const int64_t way = (int64_t)blockIdx.x * WAYS + wy;
    const bool active = wy < WAYS && way < n_ways;
    V *S = reinterpret_cast<V *>(smem_raw + (size_t)O * ps.n_mom * kProjThreads * 16) +
           (wy < WAYS ? wy : 0) * per_way;  // [B][nrow][NXI]
    V *Q = S + B * nent;                    // [B][3][NJS]
    V *Ph = Q + B * 3 * NJS;                // [B][n_x]
    const int asplit = nrow / 6;            // pairs of spins
    const int ch = (int)(way % n_chunks), a2 = (int)(way / n_chunks % asplit);
    const int64_t slab = way / n_chunks / asplit;
    const int v3 = F.lx * F.ly * F.lz;
    const int c0 = (int)((int64_t)v3 * ch / n_chunks), c1 = active ? (int)((int64_t)v3 * (ch + 1) / n_chunks) : c0;
    const int64_t base = slab / F.n_t * F.stride_cfg + (F.t0 + slab % F.n_t) * F.stride_t;
    const int js = tw % NJS, i0 = tw / NJS * I;
    Sum line[NX][O];
#pragma unroll
    for (int k = 0; k < NX; ++k)
#pragma unroll
        for (int o = 0; o < O; ++o) line[k][o].zero();
    for (int o = 0; o < O * ps.n_mom; ++o) out[o * kProjThreads].zero();
    const int n_batches = ((v3 + n_chunks - 1) / n_chunks + B - 1) / B;  // of the longest chunk
    // a thread loads the same entries of every batch, one batch ahead
    constexpr int NL = (B * (NXI == 12 ? 144 : 36) + WAY - 1) / WAY;
    int ent_b[NL], ent_off[NL];
    V pre[NL], pre_ph{0, 0};
#pragma unroll
    for (int l = 0; l < NL; ++l) {
        const int e = tw + l * WAY;
        ent_b[l] = active && e < B * nent ? e / nent : B;
        ent_off[l] = e < B * nent ? tile_index(F, e % nent, NXI) : 0;
    }
    const bool ph_lane = active && tw < B * ps.n_x;
    const int ph_b = tw / ps.n_x, ph_col = ph_lane ? ps.xcol[tw % ps.n_x] : 0;
    auto fetch = [&](int s0) {
#pragma unroll
        for (int l = 0; l < NL; ++l) {
            const int site = s0 + ent_b[l];
            double2 v = make_double2(0.0, 0.0);
            if (ent_b[l] < B && site < c1) v = load_prop(F, base + (int64_t)site * site_elems(F), ent_off[l]);
            pre[l] = V{(R)v.x, (R)v.y};
        }
        if (ph_lane && s0 + ph_b < c1) {
            const double2 v = __ldg(xtab + (int64_t)((s0 + ph_b) % F.lx) * n_dx + ph_col);
            pre_ph = Sum::first(*reinterpret_cast<const Phase *>(&v));
        }
    };
    // the thread's diquark entries: pair (x2, x3) = js, colours and sites in turn
    int x3 = 0;
    while ((x3 + 1) * (x3 + 2) / 2 <= js) ++x3;
    const int x2 = js - x3 * (x3 + 1) / 2;
    fetch(c0);
    int x = c0 % F.lx, ln = c0 / F.lx;  // of the next site
    for (int bt = 0; bt < n_batches; ++bt) {
        const int s0 = c0 + bt * B;
        __syncthreads();  // the previous batch is consumed
#pragma unroll
        for (int l = 0; l < NL; ++l)
            if (ent_b[l] < B) S[tw + l * WAY] = pre[l];
        if (ph_lane) Ph[ph_b * kProjMoms + tw % ps.n_x] = pre_ph;
        __syncthreads();
        fetch(s0 + B);
        if (active)
            for (int q = tw / NJS; q < 3 * B; q += WAY / NJS) {
                const int c = q % 3, r2 = (c + 1) % 3 * NXI, r3 = (c + 2) % 3 * NXI;
                V acc{0, 0};
                for (int g = 0; g < n_g2; g += 2) {  // spins (g, g + 1): entries -1 and +1 of C gamma_5
                    const V *lo = S + q / 3 * nent + 3 * g * NXI, *hi = lo + 3 * NXI;
                    acc = cfms(lo[r2 + x2], hi[r3 + x3], acc);
                    acc = cfma(lo[r3 + x2], hi[r2 + x3], acc);
                    acc = cfma(hi[r2 + x2], lo[r3 + x3], acc);
                    acc = cfms(hi[r3 + x2], lo[r2 + x3], acc);
                }
                Q[q * NJS + js] = acc;
            }
        __syncthreads();
        if (!active) continue;
        for (int b = 0; b < B && s0 + b < c1; ++b) {
            V g[O];
#pragma unroll
            for (int o = 0; o < O; ++o) g[o] = V{0, 0};
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                const V q = Q[(b * 3 + c) * NJS + js];
#pragma unroll
                for (int al = 0; al < 2; ++al) {
                    const V *row = S + b * nent + (3 * (2 * a2 + al) + c) * NXI + i0;
                    V r[I];
                    if constexpr (sizeof(V) == 8 && I == 2) {  // one 16-byte broadcast (rows of 96 B, i0 even)
                        const float4 w = *reinterpret_cast<const float4 *>(row);
                        r[0] = V{w.x, w.y};
                        r[1] = V{w.z, w.w};
                    } else {
#pragma unroll
                        for (int o = 0; o < I; ++o) r[o] = row[o];
                    }
#pragma unroll
                    for (int o = 0; o < I; ++o) g[al * I + o] = cfma(r[o], q, g[al * I + o]);
                }
            }
#pragma unroll
            for (int k = 0; k < NX; ++k)
                if (k < ps.n_x) {
                    if (ps.trivial[k]) {
#pragma unroll
                        for (int o = 0; o < O; ++o) line[k][o].add(g[o]);
                    } else {
                        const V ph = Ph[b * kProjMoms + k];
#pragma unroll
                        for (int o = 0; o < O; ++o) line[k][o].add(ph, g[o]);
                    }
                }
            if (++x == F.lx || s0 + b == c1 - 1) {  // end of a line: into the momenta
                const double2 *yt = ytab + (int64_t)ln * n_mom + ps.q0;
                x = 0;
                ++ln;
#pragma unroll
                for (int k = 0; k < NX; ++k) {
                    for (int m = 0; m < ps.n_mom; ++m) {
                        if (ps.nx_of[m] != k) continue;
                        const double2 p = __ldg(yt + m);
                        const Phase ph = *reinterpret_cast<const Phase *>(&p);
                        Total *t = out + m * O * kProjThreads;
#pragma unroll
                        for (int o = 0; o < O; ++o) {
                            Total v = t[o * kProjThreads];
                            v.add(ph, ps.flat[m], line[k][o]);
                            t[o * kProjThreads] = v;
                        }
                    }
#pragma unroll
                    for (int o = 0; o < O; ++o) line[k][o].zero();
                }
            }
        }
    }
    if (!active) return;
    // partial[slab][chunk][mom][(alpha, i)][js]
    const int64_t G = (int64_t)(nrow / 3) * NXI * NJS;
    for (int m = 0; m < ps.n_mom; ++m)
#pragma unroll
        for (int o = 0; o < O; ++o)
            partial[((slab * n_chunks + ch) * n_mom + ps.q0 + m) * G +
                    (int64_t)((2 * a2 + o / I) * NXI + i0 + o % I) * NJS + js] =
                out[(m * O + o) * kProjThreads].value();
}

// Pf[slab][mom][block entry]: chunk sums in order, then f = g[i; j s] - g[j; i s].
// amax (mixed): per (slab, group of n_k momenta) the bits of the largest |re| or
// |im| (nonnegative doubles order as integers); cleared before.
__global__ void __launch_bounds__(256) k_project_sum(const double2 *__restrict__ partial, int64_t n_slabs, int n_chunks,
                                                     int n_mom, int n_k, int nxi, int bs, double2 *__restrict__ Pf,
                                                     unsigned long long *__restrict__ amax) {
    const int njs = proj_njs(nxi), npair = nxi * (nxi - 1) / 2;
    const int64_t G = (int64_t)bs / (npair * nxi) * nxi * njs;
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t sm = blockIdx.y;  // slab * n_mom + mom
    double big = 0.0;
    if (e < bs) {
        const int al = e / (npair * nxi), pr = e / nxi % npair, s = e % nxi;
        const int i = c_pair_i[pr], j = c_pair_j[pr];
        const int tj = j <= s ? s * (s + 1) / 2 + j : j * (j + 1) / 2 + s;
        const int ti = i <= s ? s * (s + 1) / 2 + i : i * (i + 1) / 2 + s;
        const double2 *p = partial + (sm / n_mom * n_chunks * n_mom + sm % n_mom) * G;
        const double2 *pi = p + (int64_t)(al * nxi + i) * njs + tj, *pj = p + (int64_t)(al * nxi + j) * njs + ti;
        double2 a = make_double2(0.0, 0.0), b = a;
#pragma unroll 4
        for (int k = 0; k < n_chunks; ++k) {
            a = cadd(a, __ldg(pi + (int64_t)k * n_mom * G));
            b = cadd(b, __ldg(pj + (int64_t)k * n_mom * G));
        }
        const double2 f = csub(a, b);
        Pf[sm * bs + e] = f;
        big = fmax(fabs(f.x), fabs(f.y));
    }
    if (!amax) return;
    for (int off = 16; off > 0; off >>= 1) big = fmax(big, __shfl_xor_sync(0xffffffffu, big, off));
    if ((threadIdx.x & 31) == 0) {
        const int64_t item = sm / n_mom * (n_mom / n_k) + sm % n_mom / n_k;
        atomicMax(amax + item, (unsigned long long)__double_as_longlong(big));
    }
}

// Summed blocks of the wave's items -> wave layout (wave_index); thread = (block
// entry, item). An item is (slab, group of n_k momenta); with n_k sink functions
// (Sec. 6) the sink index of the item's block is psi = n_k * alpha + k, and block
// entry (psi; pair, single) is entry (alpha; pair, single) of the block projected
// with momentum k of the group. Pf: [slab][momentum][block] with bs_site entries
// (one sink function).
template <class Tr>
__global__ void __launch_bounds__(256) k_load_proj_blocks(const double2 *__restrict__ Pf, int64_t n_items,
                                                          int64_t item0, int W, int bs_site, int per_spin, int n_k,
                                                          int n_mom, const unsigned long long *__restrict__ amax, int T,
                                                          typename Tr::V *__restrict__ f, int32_t *__restrict__ sexp) {
    const int block_size = bs_site * n_k;
    const int n_groups = n_mom / n_k;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < (int64_t)block_size * W;
         i += (int64_t)gridDim.x * blockDim.x) {
        const int e = (int)(i % block_size), col = (int)(i / block_size);
        const int64_t item = item0 + col;
        double2 v = make_double2(0.0, 0.0);
        int se = 0;
        if (item < n_items) {
            const int64_t slab = item / n_groups;
            const int q0 = (int)(item % n_groups) * n_k;
            const int psi = e / per_spin, r = e % per_spin;
            v = Pf[(slab * n_mom + q0 + psi % n_k) * bs_site + psi / n_k * per_spin + r];
            if (amax) {
                const double big = __longlong_as_double((long long)amax[item]);
                se = big > 0.0 ? -ilogb(big) : 0;
                v = make_double2(scalbn(v.x, se), scalbn(v.y, se));
            }
        }
        Tr::wave_st(f, wave_index(e, col, T, block_size), Tr::from_d(v));
        if (e == 0) sexp[col] = se;
    }
}

// out[cfg][list][t - t0][mom][comp_stride] = C[comp][item] for the wave's items
// (n_mom: items per slab)
__global__ void k_write_items(const double2 *__restrict__ C, int64_t n_items, int64_t item0, int W, int n_comp,
                              int n_mom, int n_t, int list_idx, int n_lists, int comp_stride, double2 *out) {
    const int64_t total = (int64_t)n_comp * W;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x) {
        const int c = (int)(i / W), col = (int)(i % W);
        const int64_t item = item0 + col;
        if (item >= n_items) continue;
        const int64_t slab = item / n_mom;
        const int q = (int)(item % n_mom);
        const int cfg = (int)(slab / n_t), tt = (int)(slab % n_t);
        out[((((int64_t)cfg * n_lists + list_idx) * n_t + tt) * n_mom + q) * comp_stride + c] = C[i];
    }
}

}  // namespace mbc
