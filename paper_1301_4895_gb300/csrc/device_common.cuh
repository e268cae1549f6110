// Device helpers shared by the contraction kernels: the FP64 storage type and
// accumulator, sign flips without arithmetic, complex helpers and the
// baryon-block formulas. The mixed-precision types live in mixed_common.cuh.
#pragma once

#include <cuda_runtime.h>
#include <cstdint>

namespace mbc {

// plain complex helpers in the storage type (block construction)
__device__ __forceinline__ double2 cmul(double2 a, double2 b) {
    return make_double2(__fma_rn(a.x, b.x, -a.y * b.y), __fma_rn(a.x, b.y, a.y * b.x));
}
__device__ __forceinline__ float2 cmul(float2 a, float2 b) {
    return make_float2(__fmaf_rn(a.x, b.x, -a.y * b.y), __fmaf_rn(a.x, b.y, a.y * b.x));
}
__device__ __forceinline__ double2 cadd(double2 a, double2 b) { return make_double2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ float2 cadd(float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ double2 csub(double2 a, double2 b) { return make_double2(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ float2 csub(float2 a, float2 b) { return make_float2(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ double2 cfma(double2 a, double2 b, double2 c) {
    return make_double2(__fma_rn(a.x, b.x, __fma_rn(-a.y, b.y, c.x)), __fma_rn(a.x, b.y, __fma_rn(a.y, b.x, c.y)));
}
__device__ __forceinline__ float2 cfma(float2 a, float2 b, float2 c) {
    return make_float2(__fmaf_rn(a.x, b.x, __fmaf_rn(-a.y, b.y, c.x)), __fmaf_rn(a.x, b.y, __fmaf_rn(a.y, b.x, c.y)));
}
// c - a * b with fused multiply-adds only
__device__ __forceinline__ double2 cfms(double2 a, double2 b, double2 c) {
    return make_double2(__fma_rn(-a.x, b.x, __fma_rn(a.y, b.y, c.x)), __fma_rn(-a.x, b.y, __fma_rn(-a.y, b.x, c.y)));
}
__device__ __forceinline__ float2 cfms(float2 a, float2 b, float2 c) {
    return make_float2(__fmaf_rn(-a.x, b.x, __fmaf_rn(a.y, b.y, c.x)), __fmaf_rn(-a.x, b.y, __fmaf_rn(-a.y, b.x, c.y)));
}

// ---- precision traits ------------------------------------------------------

struct FP64Traits {
    using V = double2;  // stored stage value
    struct Acc {
        double re, im;
        __device__ __forceinline__ void zero() { re = 0.0; im = 0.0; }
        // acc += (sign) * x * y  - four DFMA, the sign flips x by bit ops
        __device__ __forceinline__ void fma(double2 x, double2 y, uint32_t neg) {
            double xr = __hiloint2double(__double2hiint(x.x) ^ (int)neg, __double2loint(x.x));
            double xi = __hiloint2double(__double2hiint(x.y) ^ (int)neg, __double2loint(x.y));
            re = __fma_rn(xr, y.x, re);
            re = __fma_rn(-xi, y.y, re);
            im = __fma_rn(xr, y.y, im);
            im = __fma_rn(xi, y.x, im);
        }
        __device__ __forceinline__ void add_shfl(unsigned mask, int off) {
            re += __shfl_xor_sync(mask, re, off);
            im += __shfl_xor_sync(mask, im, off);
        }
        __device__ __forceinline__ double2 value() const { return make_double2(re, im); }
        __device__ __forceinline__ V store() const { return make_double2(re, im); }
    };
    __device__ __forceinline__ static double2 to_d(V v) { return v; }
    __device__ __forceinline__ static V from_d(double2 v) { return v; }
    // block construction: diquarks are kept and products summed as they are
    using Q = double2;
    struct BlockAcc {
        double2 v;
        __device__ __forceinline__ void zero() { v = make_double2(0.0, 0.0); }
        __device__ __forceinline__ void add(double2 a, double2 b) { v = cfma(a, b, v); }
        __device__ __forceinline__ void sub(double2 a, double2 b) { v = cfms(a, b, v); }
        __device__ __forceinline__ Q q() const { return v; }
        __device__ __forceinline__ V block() const { return v; }
    };
    // entry idx of a wave buffer ([component][site], plain)
    __device__ __forceinline__ static V wave_ld(const V *p, int64_t idx) { return p[idx]; }
    __device__ __forceinline__ static void wave_st(V *p, int64_t idx, V v) { p[idx] = v; }
};

// ---- the G tensor (eq. def_g) in factorised form -----------------------------
// colex pair decoding for up to 24 quark index values (two relativistic
// sources): pair rank -> (i < j)
__constant__ uint8_t c_pair_i[276];
__constant__ uint8_t c_pair_j[276];

// Diquark Q[c][x2][x3] = sum_{Gamma_2, eps} v eps S[3 s2 + c2][x2] S[3 s3 + c3][x3]
// (the slot-2/slot-3 part of a block, Sec. 2) of a tile with rows at(row, column):
// spins (g, g + 1) carry the entries -1 and +1 of C gamma_5.
template <class Acc, class At>
__device__ __forceinline__ Acc diquark(At &&at, int n_g2, int c, int x2, int x3) {
    Acc acc;
    acc.zero();
    const int c2 = c == 2 ? 0 : c + 1, c3 = c == 0 ? 2 : c - 1;
    for (int g = 0; g < n_g2; g += 2) {
        const int lo = 3 * g, hi = lo + 3;
        acc.sub(at(lo + c2, x2), at(hi + c3, x3));
        acc.add(at(lo + c3, x2), at(hi + c2, x3));
        acc.add(at(hi + c2, x2), at(lo + c3, x3));
        acc.sub(at(hi + c3, x2), at(lo + c2, x3));
    }
    return acc;
}

}  // namespace mbc
