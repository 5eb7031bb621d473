// Block fixed-point arithmetic of the FP64 path (k_stage, esdg_kernels.cuh).
//
// The FP64 pipe of sm_103a takes a warp instruction every 64 cycles and
// scheduler (76 measured for a chain of DFMAs), the integer pipes one every
// two: a signed 32 x 32 + 64 bit multiply-add (IMAD.WIDE) measures at most 8.7
// cycles.  Sums of products whose operands share a scale therefore run as
// integers: a value x with |x| < 2^X becomes round(x 2^(bits - X)), bits = 57 or
// 58, in two limbs hi 2^28 + lo (lo the signed low 28 bits), a product is
// hi hi' 2^56 + (hi lo' + lo hi') 2^28 (three IMAD.WIDE into two 64-bit sums;
// lo lo' is below the last bit kept).  The scales are the
// binary exponents of the largest value of an element (per field, taken at run
// time) and of the largest absolute row sum of an element's operator (host), so
// that no sum can overflow.  In units of 2^56 of the operands' product, of which the
// two scales' product has 2^60, a sum of n products is off by the operands' rounding (to
// half of their last bit: 2 units for the values, 2 n for the operator's entries) and by
// n / 4 + 1 units of dropped low products and flooring: 100 units, 2^-53 of the scales'
// product, where all of the n <= 43 terms of a row err to one side, some ten, 2^-57,
// where the signs are mixed.  T is rounded once more (fx_pair_t).  The FP64 evaluation
// rounds every term and partial sum to 53 bits, relative to each term instead of to the
// element's largest: entries whose terms are all far below it are better there, and
// norms over an element are not.  Infinities and NaN (exponent 0x7ff) are passed on
// as NaN.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>
#include <string.h>

namespace esdg {

constexpr int FX_LO = 28;            // bits of the low limb
constexpr int FX_NONFINITE = 0x7ff;  // exponent field of infinities and NaN

// two 64-bit sums of a product sum: value (hh 2^28 + mid) 2^28
struct FxSum {
    long long hh, mid;
};

__host__ __device__ inline int2 fx_limbs(long long a) {
    const int lo = (int)((uint32_t)a << (32 - FX_LO)) >> (32 - FX_LO);
    return make_int2(lo, (int)((a - lo) >> FX_LO));
}

// the bits of a double and back (on the host too, for the tests)
__host__ __device__ __forceinline__ long long fx_bits(double x) {
#ifdef __CUDA_ARCH__
    return __double_as_longlong(x);
#else
    long long i;
    memcpy(&i, &x, 8);
    return i;
#endif
}
__host__ __device__ __forceinline__ double fx_double(long long i) {
#ifdef __CUDA_ARCH__
    return __longlong_as_double(i);
#else
    double x;
    memcpy(&x, &i, 8);
    return x;
#endif
}

__host__ __device__ __forceinline__ int fx_hi(double x) {
#ifdef __CUDA_ARCH__
    return __double2hiint(x);
#else
    return (int)(fx_bits(x) >> 32);
#endif
}
__host__ __device__ __forceinline__ uint32_t fx_lo(double x) {
#ifdef __CUDA_ARCH__
    return (uint32_t)__double2loint(x);
#else
    return (uint32_t)fx_bits(x);
#endif
}

// The larger of two values >= 0, on the integer pipes; NaN if one is NaN, of either
// sign (the square root of a negative depth has the sign bit set).
__host__ __device__ __forceinline__ double r_max_nonneg(double a, double b) {
    const long long x = fx_bits(a) & 0x7fffffffffffffffll, y = fx_bits(b) & 0x7fffffffffffffffll;
    return fx_double(x > y ? x : y);
}

// exponent field of x
__host__ __device__ __forceinline__ int fx_exp(double x) { return (fx_hi(x) >> 20) & 0x7ff; }
// largest exponent field of the warp as the X of |x| < 2^X
__device__ __forceinline__ int fx_max(int e) { return __reduce_max_sync(0xffffffffu, e); }
__host__ __device__ __forceinline__ int fx_scale(int emax) { return emax - 1022; }

// round(x 2^(BITS - X)) for |x| < 2^X (X = fx_scale of an exponent field at
// least x's), ties away from zero.
template <int BITS>
__host__ __device__ __forceinline__ long long fx_from(double x, int X) {
    const int hi = fx_hi(x);
    const int e = (hi >> 20) & 0x7ff;
    // mantissa 2^10 (63 bits; zeros and subnormals: no leading bit, exponent 1), to
    // be shifted down by d >= 62 - BITS
    const uint32_t mh = ((uint32_t)hi & 0xfffffu) | (e ? 0x100000u : 0u);
    const uint64_t m = (((uint64_t)mh << 32) | fx_lo(x)) << 10;
    const int d = (63 - BITS) + (X + 1022 - max(e, 1));
    const uint64_t v = ((m >> min(d - 1, 63)) + 1) >> 1;
    return hi < 0 ? -(long long)v : (long long)v;
}

// s 2^sh as a double (round to nearest, ties away from zero).  ALL: also outside the
// normal range (subnormal below it, infinite above).
template <bool ALL>
__host__ __device__ __forceinline__ double fx_to_(long long s, int sh) {
    const uint64_t a = (uint64_t)(s < 0 ? -s : s);
#ifdef __CUDA_ARCH__
    const int lz = __clzll((long long)a);
#else
    const int lz = a ? __builtin_clzll(a) : 64;
#endif
    const uint64_t y = a << (lz & 63);
    const uint64_t r = (y >> 11) + ((y >> 10) & 1u);  // 2^52 .. 2^53
    const int E = sh - lz + 1086;                      // exponent field
    uint64_t bits = (((uint64_t)(uint32_t)(E - 1)) << 52) + r;
    if (ALL && (unsigned)(E - 1) >= 2046u)
        bits = E > 0 ? 0x7ff0000000000000ull : E < -52 ? 0 : ((y >> (11 - E)) + 1) >> 1;
    if (a == 0) bits = 0;
    return fx_double((long long)(bits | (s < 0 ? 0x8000000000000000ull : 0ull)));
}
// n values x[i] = s[i] 2^sh(i).  The integers s[i] other than 0 have sizes from 1 to 2^63,
// so the scales alone say whether all results lie in the normal range (1 <= sh + 1023,
// sh + 1085 <= 2046); the whole group takes one branch where they do not (in line the
// shift that the others need cost every sum 1.5%, a test of each result 1%).
template <int n, typename Sh>
__host__ __device__ __forceinline__ void fx_to(const long long* s, Sh sh, double* x) {
    bool inside = true;
#pragma unroll
    for (int i = 0; i < n; ++i) inside &= (unsigned)(sh(i) + 1022) <= 1983u;
    if (__builtin_expect(!inside, 0)) {
#pragma unroll
        for (int i = 0; i < n; ++i) x[i] = fx_to_<true>(s[i], sh(i));
    } else {
#pragma unroll
        for (int i = 0; i < n; ++i) x[i] = fx_to_<false>(s[i], sh(i));
    }
}

__host__ __device__ __forceinline__ void fx_mac(FxSum& s, int2 a, int2 b) {
    s.hh += (long long)a.y * b.y;
    s.mid += (long long)a.x * b.y;
    s.mid += (long long)a.y * b.x;
}
// the sum in units of 2^56 of the operands' product
__host__ __device__ __forceinline__ long long fx_value(const FxSum& s) { return s.hh + (s.mid >> FX_LO); }
__host__ __device__ __forceinline__ int2 fx_neg(int2 a) { return make_int2(-a.x, -a.y); }
__device__ __forceinline__ int2 fx_shfl(int2 a, int src) {
    return make_int2(__shfl_sync(0xffffffffu, a.x, src), __shfl_sync(0xffffffffu, a.y, src));
}

// Operand widths.  Pair terms: momenta hu, hv 57 bits (their pair sums 58),
// velocities and free surface 58, the stored operator's largest row sums of
// |Qx| and of |Qy| 59 each (a scale each: on a stretched element one is far below
// the other) with entries of at most 58 (a row's entries of Qx and of Qy
// sum to zero, so none exceeds half the row's); T in units of 2^-57 of its scale.
// Contractions: values 58, the operator's largest row sum 58.
constexpr int FX_MOM = 57, FX_VAL = 58, FX_PAIR = 59, FX_ROW = 58, FX_T = 57;

// Two scales in one word (an element's XQx and XQy).
__host__ __device__ inline int fx_pack(int x, int y) { return (int)((uint32_t)y << 16 | ((uint32_t)x & 0xffffu)); }
__host__ __device__ inline int fx_pack_x(int w) { return (int)(int16_t)(w & 0xffff); }
__host__ __device__ inline int fx_pack_y(int w) { return w >> 16; }

// The two products of T on one scale XT: the momenta take the scales that give
// both XT, so that the sum needs no shift; the smaller product loses the bits
// that are below the larger one's last.
__host__ __device__ __forceinline__ int fx_align(int XQx, int XQy, int& Xhu, int& Xhv) {
    const int XT = max(XQx + Xhu, XQy + Xhv);
    Xhu = XT - XQx;
    Xhv = XT - XQy;
    return XT;
}

// T = Qx (hu_l + hu_m) + Qy (hv_l + hv_m): T 2^(57 - XT), off by at most 3/4 besides the
// operands' rounding (its own half, the low products' and the floor's eighth each)
__host__ __device__ __forceinline__ long long fx_pair_t(int2 qx, int2 qy, int2 hu, int2 hv) {
    FxSum s;
    s.hh = (long long)qx.y * hu.y;
    s.mid = (long long)qx.x * hu.y;
    s.mid += (long long)qx.y * hu.x;
    fx_mac(s, qy, hv);
    return (fx_value(s) + 4) >> 3;
}

}  // namespace esdg
