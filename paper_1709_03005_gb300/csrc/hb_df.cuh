// Double-float arithmetic on the FP32 pipes: a value is an unevaluated sum
// hi + lo of two floats (about 48 significant bits).  The error-free
// transformations are Knuth's TwoSum and the FMA product error
// (Dekker / Ogita-Rump-Oishi); the conversion back to FP64 uses integer
// operations only, because the FP64 pipe of this part is slow.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace hb {

// Sums as FMAs with a factor of one that the compiler cannot see: an FMA and
// an addition give the same bits, but a chain of both kinds runs at 0.6 of the
// rate of FMAs alone (5.8 df_fma per SM and clock against 9.0; in f32x2
// instructions, two sums at a time, 9.7).
static __constant__ float kOne = 1.0f;
__device__ __forceinline__ float f_add(float a, float b) { return __fmaf_rn(a, kOne, b); }
__device__ __forceinline__ float f_sub(float a, float b) { return __fmaf_rn(b, -kOne, a); }

// s + e = a + b exactly
__device__ __forceinline__ void df_two_sum(float a, float b, float &s, float &e) {
    s = f_add(a, b);
    const float bp = f_sub(s, a);
    e = f_add(f_sub(a, f_sub(s, bp)), f_sub(b, bp));
}

// (hi, lo) := (ah, al) + (bh, bl), renormalised
__device__ __forceinline__ void df_add2(float &hi, float &lo, float bh, float bl) {
    float s, e;
    df_two_sum(hi, bh, s, e);
    e = f_add(e, f_add(lo, bl));
    hi = f_add(s, e);
    lo = f_sub(e, f_sub(hi, s));
}

// hi + lo as a double, with integer operations only.  Both are aligned into a
// 64-bit integer with 38 bits of headroom below the larger exponent, added
// exactly, and the result is truncated to 53 bits (relative error below
// 2^-52).  FP32 subnormals are treated as zero.
__device__ __forceinline__ double df_to_double(float hi, float lo) {
    const uint32_t bh = __float_as_uint(hi), bl = __float_as_uint(lo);
    const int eh = (int)((bh >> 23) & 0xFF), el = (int)((bl >> 23) & 0xFF);
    long long mh = eh ? (long long)((bh & 0x7FFFFFu) | 0x800000u) : 0;
    long long ml = el ? (long long)((bl & 0x7FFFFFu) | 0x800000u) : 0;
    if (bh >> 31) mh = -mh;
    if (bl >> 31) ml = -ml;
    const int base = eh > el ? eh : el;
    // value = (mh 2^(eh-base) + ml 2^(el-base)) * 2^(base - 150)
    const int sh_h = 38 - (base - eh), sh_l = 38 - (base - el);
    long long acc = 0;
    if (mh) acc += sh_h >= 0 ? (mh << sh_h) : (sh_h > -63 ? (mh >> -sh_h) : 0);
    if (ml) acc += sh_l >= 0 ? (ml << sh_l) : (sh_l > -63 ? (ml >> -sh_l) : 0);
    if (acc == 0) return 0.0;
    const unsigned long long neg = acc < 0 ? 1ull : 0ull;
    unsigned long long u = neg ? (unsigned long long)(-acc) : (unsigned long long)acc;
    const int lz = __clzll((long long)u);            // leading zeros, u > 0
    const int top = 63 - lz;                          // position of the leading one
    // normalise to 53 bits: leading one at bit 52
    if (top > 52) u >>= (top - 52);
    else u <<= (52 - top);
    // exponent: value = u * 2^(top - 52) * 2^(base - 150 - 38), u in [2^52, 2^53)
    const int e2 = top + base - 150 - 38;             // unbiased exponent of the leading one
    const long long be = (long long)e2 + 1023;
    if (be <= 0) return 0.0;                          // below the FP64 normal range
    const unsigned long long bits = (neg << 63) | ((unsigned long long)be << 52) | (u & 0xFFFFFFFFFFFFFull);
    return __longlong_as_double((long long)bits);
}

// A float as a double, from its bits (FP32 subnormals give zero, infinities and
// NaNs their like).
__device__ __forceinline__ double float_bits_to_double(float x) {
    const uint32_t u = __float_as_uint(x), m = u & 0x7FFFFFFFu;
    uint32_t hi = (m >> 3) + 0x38000000u;
    hi = m < 0x00800000u ? 0u : (m >= 0x7F800000u ? (hi | 0x7FF00000u) : hi);
    return __hiloint2double((int)(hi | (u & 0x80000000u)), m < 0x00800000u ? 0 : (int)(u << 29));
}

// hi + lo as a double where one FP64 addition can be afforded: a tenth of the
// instructions of df_to_double, correctly rounded.
__device__ __forceinline__ double df_sum(float hi, float lo) {
    return float_bits_to_double(hi) + float_bits_to_double(lo);
}

// Sum accumulators with one interface: add / subtract table entry i, where a
// table exists as FP64 and as (hi, lo) float pairs.  AccD sums the FP64 table
// on the FP64 pipe; AccF sums the float pairs in double-float.
struct AccD {
    double v = 0.0;
    using Entry = double;
    static __device__ __forceinline__ Entry entry(const double *t, const float2 *, int64_t i) { return __ldg(t + i); }
    __device__ __forceinline__ void add_entry(Entry x) { v += x; }
    __device__ __forceinline__ void sub_entry(Entry x) { v -= x; }
    __device__ __forceinline__ void add(const double *t, const float2 *, int64_t i) { v += __ldg(t + i); }
    __device__ __forceinline__ void sub(const double *t, const float2 *, int64_t i) { v -= __ldg(t + i); }
    __device__ __forceinline__ void neg() { v = -v; }
    __device__ __forceinline__ void add_const(double c) { v += c; }
    __device__ __forceinline__ double value() const { return v; }
};

struct AccF {
    float h = 0.0f, l = 0.0f;
    using Entry = float2;
    static __device__ __forceinline__ Entry entry(const double *, const float2 *t, int64_t i) { return __ldg(t + i); }
    __device__ __forceinline__ void add_entry(Entry x) { df_add2(h, l, x.x, x.y); }
    __device__ __forceinline__ void sub_entry(Entry x) { df_add2(h, l, -x.x, -x.y); }
    __device__ __forceinline__ void add(const double *, const float2 *t, int64_t i) {
        const float2 x = __ldg(t + i);
        df_add2(h, l, x.x, x.y);
    }
    __device__ __forceinline__ void sub(const double *, const float2 *t, int64_t i) {
        const float2 x = __ldg(t + i);
        df_add2(h, l, -x.x, -x.y);
    }
    __device__ __forceinline__ void neg() { h = -h; l = -l; }
    __device__ __forceinline__ void add_const(double c) {   // host-side constants only (e_core)
        const float ch = (float)c;
        df_add2(h, l, ch, (float)(c - (double)ch));
    }
    __device__ __forceinline__ double value() const { return df_to_double(h, l); }
};

// (hi, lo) += a * b for double-float a, b (products exact by FMA, TwoSum on the
// high words; the low words collect the rest)
__device__ __forceinline__ void df_fma(float &hi, float &lo, float ah, float al, float bh, float bl) {
    const float ph = ah * bh;
    const float pe = fmaf(ah, bh, -ph);
    const float pl = fmaf(ah, bl, fmaf(al, bh, pe));
    float s, e;
    df_two_sum(hi, ph, s, e);
    hi = s;
    lo = f_add(lo, f_add(e, pl));
}

// renormalise (hi, lo) so that |lo| <= ulp(hi) / 2
__device__ __forceinline__ void df_norm(float &hi, float &lo) {
    const float s = f_add(hi, lo);
    lo = f_sub(lo, f_sub(s, hi));
    hi = s;
}

// Two floats in a register pair, and their f32x2 instructions (each half rounded
// as the single instruction rounds it).
struct f2 { unsigned long long v; };
__device__ __forceinline__ f2 f2_pack(float a, float b) {
    f2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ void f2_unpack(f2 x, float &a, float &b) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(x.v));
}
__device__ __forceinline__ f2 f2_add(f2 a, f2 b) {
    f2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ f2 f2_sub(f2 a, f2 b) {
    f2 r;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ f2 f2_mul(f2 a, f2 b) {
    f2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ f2 f2_fma(f2 a, f2 b, f2 c) {
    f2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
    return r;
}

// df_fma for two sums at a time, to the same bits; nah = -ah, so that the
// product's error needs no negation of the product.
__device__ __forceinline__ void df_fma(f2 &hi, f2 &lo, f2 ah, f2 nah, f2 al, f2 bh, f2 bl) {
    const f2 nph = f2_mul(nah, bh);
    const f2 pl = f2_fma(ah, bl, f2_fma(al, bh, f2_fma(ah, bh, nph)));
    const f2 s = f2_sub(hi, nph), bp = f2_sub(s, hi);
    const f2 e = f2_sub(f2_sub(hi, f2_sub(s, bp)), f2_add(nph, bp));
    hi = s;
    lo = f2_add(lo, f2_add(e, pl));
}

// (hi, lo) += x for two sums: TwoSum on the high words
__device__ __forceinline__ void df_add(f2 &hi, f2 &lo, f2 x) {
    const f2 s = f2_add(hi, x), bp = f2_sub(s, hi);
    lo = f2_add(lo, f2_add(f2_sub(hi, f2_sub(s, bp)), f2_sub(x, bp)));
    hi = s;
}

__device__ __forceinline__ void df_norm(f2 &hi, f2 &lo) {
    const f2 s = f2_add(hi, lo);
    lo = f2_sub(lo, f2_sub(s, hi));
    hi = s;
}

// FP64 array -> (hi, lo) float pairs, hi = x rounded to float, lo = the rest
// rounded to float (|x - hi - lo| <= 2^-48 |x| for x in the float range).
void split_df(const double *x, int64_t n, float2 *out, cudaStream_t s);

}  // namespace hb
