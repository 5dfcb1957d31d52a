// Device arithmetic of the fixed-point Krylov kernel (krylov_fixed.cu, whose header describes the
// numbers): split integers, their products and sums.
#pragma once

#include <cuda_runtime.h>

namespace elses {

// V = h 2^28 + l with |l| <= 2^27, as int2 (h, l).
__host__ __device__ __forceinline__ int2 fx_split(long long v) {
    const int h = (int)((v + (1ll << 27)) >> 28);
    return make_int2(h, (int)((unsigned)v - ((unsigned)h << 28)));
}

// Sum of products in units of 2^56: h + m / 2^28.
struct Fx {
    long long h = 0, m = 0;
};

// acc += a b. As a low product with carry into a high one, which becomes a single 64-bit
// multiply-add instruction; mad.wide.s32 compiles to a multiplication and a separate addition
// (72 products of pass A's inner loop and their loads, 8 warps: 657 clocks instead of 737).
__device__ __forceinline__ void fx_mad(long long& acc, int a, int b) {
    asm("{.reg .u32 l, h;\n\t"
        "mov.b64 {l, h}, %0;\n\t"
        "mad.lo.cc.u32 l, %1, %2, l;\n\t"
        "madc.hi.s32 h, %1, %2, h;\n\t"
        "mov.b64 %0, {l, h};}"
        : "+l"(acc)
        : "r"(a), "r"(b));
}
__device__ __forceinline__ void fx_mac(Fx& acc, const int2 a, const int2 b) {
    fx_mad(acc.h, a.x, b.x);
    fx_mad(acc.m, a.x, b.y);
    fx_mad(acc.m, a.y, b.x);
}
__device__ __forceinline__ long long fx_wide(int a, int b) {
    long long v;
    asm("mul.wide.s32 %0, %1, %2;" : "=l"(v) : "r"(a), "r"(b));
    return v;
}
__device__ __forceinline__ void fx_mul(Fx& acc, const int2 a, const int2 b) {
    acc.h = fx_wide(a.x, b.x);
    acc.m = fx_wide(a.x, b.y);
    fx_mad(acc.m, a.y, b.x);
}
// the same with the half unit by which fx_pair's truncation rounds
__device__ __forceinline__ void fx_mul_half(Fx& acc, const int2 a, const int2 b) {
    acc.h = fx_wide(a.x, b.x);
    acc.m = 1ll << 27;
    fx_mad(acc.m, a.x, b.y);
    fx_mad(acc.m, a.y, b.x);
}
__device__ __forceinline__ long long fx_fold(const Fx& a) { return a.h + ((a.m + (1ll << 27)) >> 28); }

// The sum (begun by fx_mul_half) as a split pair with 0 <= l < 2^28: fewer instructions than
// fx_split(fx_fold()). For sums below 2^58.5 (h) and 2^58.5 (m).
__device__ __forceinline__ int2 fx_pair(const Fx& a) {
    const int l = ((int)a.h & 0x0fffffff) + (int)(a.m >> 28);
    return make_int2((int)(a.h >> 28) + (l >> 28), l & 0x0fffffff);
}
__device__ __forceinline__ double fx_value(const int2 v) { return (double)(((long long)v.x << 28) + v.y); }

// Coefficients gk (lane l: values l and l + 32 of n + 1) as integers of one scale 2^eg, by one warp:
// each below 2^58, their sum below 2^60, and eg <= 60 so that the vector they are subtracted from
// (below 2^56, in units of 2^(eg - 56)) stays below 2^60; *shift = 56 - eg.
__device__ __forceinline__ void fx_coefs(const double (&gk)[2], int n, int2* g, int* shift) {
    const int lane = threadIdx.x & 31;
    const unsigned top = __reduce_max_sync(0xffffffffu, max((unsigned)__double2hiint(gk[0]) & 0x7fffffffu,
                                                            (unsigned)__double2hiint(gk[1]) & 0x7fffffffu));
    const int e = max((int)(top >> 20) - 1023, -900);           // largest |g| < 2^(e + 1)
    // the sum over 2^e, in single precision and rounded up
    const double down = __longlong_as_double((long long)(1023 - e) << 52);
    float sum = __double2float_ru(fabs(gk[0]) * down);
    if (n >= 32) sum += __double2float_ru(fabs(gk[1]) * down);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
    const int es = (int)(__float_as_uint(sum * 1.001f) >> 23) - 127 + 1;      // sum < 2^(e + es)
    const int eg = max(-900, min(60, min(57 - e, 60 - e - es)));
    const double scale = __longlong_as_double((long long)(1023 + eg) << 52);
#pragma unroll
    for (int r = 0; r < 2; ++r)
        if (32 * r <= n && lane + 32 * r <= n) g[lane + 32 * r] = fx_split(__double2ll_rn(gk[r] * scale));
    if (lane == 0) *shift = 56 - eg;
}

// ------------------------------------------------------------------------------ tensor memory
// Tensor memory as storage of the threads: 128 lanes of 512 32-bit columns; warp w of a CTA reaches
// lanes 32 (w mod 4) to + 31. A load waits for its values within the same instruction sequence.
__device__ __forceinline__ void fx_tmem_alloc(unsigned* to, int cols) {
    const unsigned at = (unsigned)__cvta_generic_to_shared(to);
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(at), "r"(cols) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void fx_tmem_free(unsigned at, int cols) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(at), "r"(cols) : "memory");
}
__device__ __forceinline__ void fx_tmem_st(unsigned at, const int4 v) {
    __syncwarp();
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1, %2, %3, %4};\n\t"
        "tcgen05.wait::st.sync.aligned;" ::"r"(at), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w) : "memory");
}
#define FX_LD(o0, o1, o2, o3, ad) "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%" #o0 ", %" #o1 ", %" #o2 ", %" #o3 "}, [%" #ad "];\n\t"
#define FX_OUT(v) "=&r"((v).x), "=&r"((v).y), "=&r"((v).z), "=&r"((v).w)
// N units, `step` columns apart
template <int N>
__device__ __forceinline__ void fx_tmem_ld(unsigned at, int step, int4 (&v)[N]) {
    __syncwarp();
    static_assert(N == 2 || N == 4, "units at a time");
    if constexpr (N == 2)
        asm volatile(FX_LD(0, 1, 2, 3, 8) FX_LD(4, 5, 6, 7, 9) "tcgen05.wait::ld.sync.aligned;"
                     : FX_OUT(v[0]), FX_OUT(v[1]) : "r"(at), "r"(at + step) : "memory");
    else
        asm volatile(FX_LD(0, 1, 2, 3, 16) FX_LD(4, 5, 6, 7, 17) FX_LD(8, 9, 10, 11, 18) FX_LD(12, 13, 14, 15, 19)
                     "tcgen05.wait::ld.sync.aligned;"
                     : FX_OUT(v[0]), FX_OUT(v[1]), FX_OUT(v[2]), FX_OUT(v[3])
                     : "r"(at), "r"(at + step), "r"(at + 2 * step), "r"(at + 3 * step) : "memory");
}
// two neighbouring units of four vectors `step` columns apart: v[kk], v[4 + kk] of vector kk
__device__ __forceinline__ void fx_tmem_ld4x2(unsigned at, int step, int4 (&v)[8]) {
    __syncwarp();
    asm volatile(FX_LD(0, 1, 2, 3, 32) FX_LD(4, 5, 6, 7, 33) FX_LD(8, 9, 10, 11, 34) FX_LD(12, 13, 14, 15, 35)
                 FX_LD(16, 17, 18, 19, 36) FX_LD(20, 21, 22, 23, 37) FX_LD(24, 25, 26, 27, 38) FX_LD(28, 29, 30, 31, 39)
                 "tcgen05.wait::ld.sync.aligned;"
                 : FX_OUT(v[0]), FX_OUT(v[1]), FX_OUT(v[2]), FX_OUT(v[3]), FX_OUT(v[4]), FX_OUT(v[5]), FX_OUT(v[6]),
                   FX_OUT(v[7])
                 : "r"(at), "r"(at + step), "r"(at + 2 * step), "r"(at + 3 * step), "r"(at + 4), "r"(at + step + 4),
                   "r"(at + 2 * step + 4), "r"(at + 3 * step + 4) : "memory");
}
#undef FX_LD
#undef FX_OUT

// v / 2^q rounded, q of either sign (|v| <= 2^56 and q >= -4 here; q > 62 gives 0)
__device__ __forceinline__ long long fx_shr(long long v, int q) {
    if (q <= 0) return v << -q;
    if (q > 62) return 0;
    return (v + (1ll << (q - 1))) >> q;
}

}  // namespace elses
