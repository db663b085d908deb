// Device helpers shared by the activation prologue and the calibration kernels: Eq. 1
// (quantization of a floating-point activation to int8) on 16 channels at a time.
#pragma once
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <math.h>
#include <stdint.h>

#include "flexiq.h"

namespace flexiq {

// Eq. 1 divides by the scale.  The scale is the same for every element, so its correctly
// rounded reciprocal r = RN(1/S) is computed once per thread and each quotient follows from
// two Newton corrections with exact fused residuals:
//     t = RN(x*r);  t = RN(t + r*(x - S*t));  t = RN(t + r*(x - S*t))
// With r correctly rounded and the first corrected t faithful, the last step yields the
// correctly rounded quotient RN(x/S) (Markstein's theorem), i.e. the IEEE division result,
// at five instructions per element.  (Only the final integer matters here: results in the
// subnormal range may differ but round to 0 either way.)  Infinite inputs, or inputs whose product with
// r overflows, turn the corrections into NaN (inf - inf); the clip's fmaxf(NaN, lo) then yields lo,
// which is right for the negative side only.  So x is first capped at 256 S from above -- every value
// beyond it quantizes to 127 anyway -- and both infinities saturate as Eq. 1's clip says.  NaN inputs
// have no place in Eq. 1; the cap replaces them too, so they quantize like +infinity, and the short forms below do the same.
struct Divider {
    float S, r, lim;
    __device__ __forceinline__ float operator()(float x) const
    {
        x = fminf(x, lim);
        float t = __fmul_rn(x, r);
        t = __fmaf_rn(__fmaf_rn(-S, t, x), r, t);
        t = __fmaf_rn(__fmaf_rn(-S, t, x), r, t);
        return t;
    }
    // lo first: the quotient of -infinity is a NaN, see above (that of a NaN input is large, the cap has replaced it)
    __device__ __forceinline__ static float clip(float t, float lo, float hi) { return fminf(fmaxf(t, lo), hi); }
};
__device__ __forceinline__ Divider make_divider(float scale)
{
    Divider d;
    d.S = scale;
    d.r = __frcp_rn(scale);
    d.lim = __fmul_rn(256.0f, scale);
    return d;
}

// The activation prologue's arithmetic has to keep up with the memory, and only the final integer matters there: q(x) =
// clip(rne(RN(x/S))) is a monotone step function of x, so any monotone form with the same steps is as exact.
//
// fp32 inputs, two operations and a conversion:
//     t = RN(x * r_hi + RN(x * r_lo)),   r_hi the largest float below 1/S, r_lo = RN(1/S - r_hi) > 0
// t = RN(x/S (1 + d)) with |d| <= 2^-46 (2^-47 from each of the two roundings of the small part, which is at
// most 2^-23 of the whole).  It rounds to another integer than RN(x/S) only where x/S lies within 2^-46 of, and not on the
// same side of, a value m where RN meets a half-integer h in [2^e, 2^(e+1)), half a unit in the last place from h.  With
// s the 24-bit integer significand of S, x - m S is, in units of half of S's last place, an integer minus or plus
// s 2^(e-23).  If 2^(23-e) divides s this is a whole number, not zero (m has 25 significant bits, x has 24), hence
// at least 2^-32 of x; otherwise it is at least |d_e| 2^(e-23), hence |d_e| 2^-49 of x, with d_e the signed distance of s
// from the nearest multiple of 2^(23-e).  So where every d_e, e = -1 .. 6, is zero or at least 9 in magnitude
// the steps are the same for every x; for the other scales (one in some 7000) the general division runs.
//
// 16-bit inputs, one operation: fma(x, r, 1.5 * 2^23), r = RN(1/S), whose low byte is the integer.  Its steps are
// compared with Eq. 1's on the host, at the two representable inputs on either side of each of the 128 half-integers
// (both forms are odd in x): the same for 99.3 % of the scales with fp16 inputs and 99.9 % with bf16; the general
// division serves the rest.
//
// Infinite x stay infinite with their sign in both forms (all factors are positive) and saturate.  NaN inputs stay NaN, which
// the clip turns into its upper bound by taking the minimum first.
constexpr float kRoundMagic = 12582912.0f;   // 1.5 * 2^23
enum QuotientForm { kQuotGeneral = 0, kQuotTwoTerm = 1, kQuotMagic = 2 };
struct TwoTerm {
    float r_hi, r_lo;
    __device__ __forceinline__ float operator()(float x) const { return __fmaf_rn(x, r_hi, __fmul_rn(x, r_lo)); }
    __device__ __forceinline__ static float clip(float t, float lo, float hi) { return fmaxf(fminf(t, hi), lo); }
};
struct QuotientPlan { int form; float r_hi, r_lo; };
inline QuotientPlan plan_quotient(float S, int dtype)
{
    QuotientPlan p{kQuotGeneral, 0.f, 0.f};
    if (!(S > 0x1p-100f && S < 0x1p100f)) return p;   // no under- or overflow below (int8 input passes any scale)
    if (dtype == FLEXIQ_DTYPE_F32) {
        int exp;
        const int s = (int)ldexpf(frexpf(S, &exp), 24);   // significand in [2^23, 2^24)
        for (int e = -1; e <= 6; ++e) {
            const int mod = 1 << (23 - e), d = s & (mod - 1);
            if (d != 0 && (d < 9 || mod - d < 9)) return p;
        }
        const double r = 1.0 / (double)S;                 // 53 bits: its error is far below the bound's slack
        p.r_hi = (float)r;
        if ((double)p.r_hi >= r) p.r_hi = nextafterf(p.r_hi, 0.f);
        p.r_lo = (float)(r - (double)p.r_hi);
        p.form = kQuotTwoTerm;
    } else if (dtype == FLEXIQ_DTYPE_F16 || dtype == FLEXIQ_DTYPE_BF16) {
        const int bits = dtype == FLEXIQ_DTYPE_F16 ? 10 : 7, emin = dtype == FLEXIQ_DTYPE_F16 ? -14 : -126;
        const double largest = dtype == FLEXIQ_DTYPE_F16 ? 65504.0 : 0x1.fep127;
        p.r_hi = (float)(1.0 / (double)S);
        int exp;
        const uint32_t s = (uint32_t)ldexpf(frexpf(S, &exp), 24);   // significand in [2^23, 2^24)
        for (int k = 0; k < 128; ++k) {
            // Both quotients are within 2^-23 of x/S (r's rounding, and RN's), so only inputs that close to (k + 1/2) S can differ.  In units
            // of half of S's last place that is v = (2k + 1) s, and the type's inputs near it are multiples of `unit` (or of more, where
            // they are subnormal): few of the 128 have one near enough, which is then looked at.
            const uint32_t v = (2u * (uint32_t)k + 1u) * s, unit = 1u << (31 - __builtin_clz(v) - bits), low = v & (unit - 1u);
            if ((low < unit - low ? low : unit - low) > (v >> 21)) continue;
            const double at = ((double)k + 0.5) * (double)S;   // exact
            const int e = ilogb(at);
            const double ulp = ldexp(1.0, (e > emin ? e : emin) - bits), below = floor(at / ulp) * ulp;
            for (int i = 0; i < 2; ++i) {
                const double x = below + i * ulp;
                if (x > largest) continue;
                if (fmaf((float)x, p.r_hi, kRoundMagic) - kRoundMagic != rintf((float)x / S)) return p;
            }
        }
        p.form = kQuotMagic;
    }
    return p;
}

// two int32 -> two saturated int8 in the low half, upper half taken from c's low half
__device__ __forceinline__ unsigned pack2_sat_s8(int hi, int lo, unsigned c)
{
    unsigned d;
    asm("cvt.pack.sat.s8.s32.b32 %0, %1, %2, %3;" : "=r"(d) : "r"(hi), "r"(lo), "r"(c));
    return d;
}
// clip(round_half_even(t), -128, 127) of four values, packed little-endian
__device__ __forceinline__ unsigned quant4(float t0, float t1, float t2, float t3)
{
    const unsigned top = pack2_sat_s8(__float2int_rn(t3), __float2int_rn(t2), 0u);
    return pack2_sat_s8(__float2int_rn(t1), __float2int_rn(t0), top);
}

// Loads the 16 channels starting at p as fp32 (exact widening for fp16 / bf16).
template <int DTYPE>
__device__ __forceinline__ void load16(const void *p, float x[16])
{
    if (DTYPE == FLEXIQ_DTYPE_F32) {
        const float4 *v = reinterpret_cast<const float4 *>(p);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const float4 f = v[i];
            x[4 * i + 0] = f.x; x[4 * i + 1] = f.y; x[4 * i + 2] = f.z; x[4 * i + 3] = f.w;
        }
    } else {
        const uint4 *v = reinterpret_cast<const uint4 *>(p);
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const uint4 u = v[i];
            const unsigned w[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                if (DTYPE == FLEXIQ_DTYPE_F16) {
                    const __half2 h = *reinterpret_cast<const __half2 *>(&w[k]);
                    x[8 * i + 2 * k] = __low2float(h);
                    x[8 * i + 2 * k + 1] = __high2float(h);
                } else {  // bf16: the 16 bits are the top half of an fp32
                    x[8 * i + 2 * k] = __uint_as_float(w[k] << 16);
                    x[8 * i + 2 * k + 1] = __uint_as_float(w[k] & 0xffff0000u);
                }
            }
        }
    }
}

// The 16 channels of one slab chunk as four words of packed int8: q = Eq. 1 of the input,
// clipped to [lo, hi] (both integers, so clipping before the rounding gives the same value
// as clipping after it).  int8 input is only clipped.
template <int DTYPE>
__device__ __forceinline__ void quantize16(const void *p, const Divider &div, float lo, float hi, unsigned w[4])
{
    if (DTYPE == FLEXIQ_DTYPE_I8) {
        const uint4 u = *reinterpret_cast<const uint4 *>(p);
        const unsigned in[4] = {u.x, u.y, u.z, u.w};
        const int ilo = (int)lo, ihi = (int)hi;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            int b[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) b[j] = max(ilo, min(ihi, (int)(signed char)((in[k] >> (8 * j)) & 0xff)));
            w[k] = pack2_sat_s8(b[1], b[0], pack2_sat_s8(b[3], b[2], 0u));
        }
    } else {
        float x[16];
        load16<DTYPE>(p, x);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            float t[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) t[j] = Divider::clip(div(x[4 * k + j]), lo, hi);
            w[k] = quant4(t[0], t[1], t[2], t[3]);
        }
    }
}

// The four channels of word k of a chunk already in registers (16-byte pieces), widened to fp32.
template <int DTYPE>
__device__ __forceinline__ void widen4(const uint4 *raw, int k, float x[4])
{
    if (DTYPE == FLEXIQ_DTYPE_F32) {
        const uint4 u = raw[k];
        x[0] = __uint_as_float(u.x); x[1] = __uint_as_float(u.y); x[2] = __uint_as_float(u.z); x[3] = __uint_as_float(u.w);
    } else {
        const uint4 u = raw[k >> 1];
        const unsigned v[2] = {(k & 1) ? u.z : u.x, (k & 1) ? u.w : u.y};
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            if (DTYPE == FLEXIQ_DTYPE_F16) {
                const __half2 h = *reinterpret_cast<const __half2 *>(&v[i]);
                x[2 * i] = __low2float(h);
                x[2 * i + 1] = __high2float(h);
            } else {  // bf16: the 16 bits are the top half of an fp32
                x[2 * i] = __uint_as_float(v[i] << 16);
                x[2 * i + 1] = __uint_as_float(v[i] & 0xffff0000u);
            }
        }
    }
}
// quantize16 for a chunk in registers, floating-point input, through the quotient `div`
template <int DTYPE, class Q>
__device__ __forceinline__ void quantize_raw(const uint4 *raw, const Q &div, float lo, float hi, unsigned w[4])
{
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        float x[4], t[4];
        widen4<DTYPE>(raw, k, x);
#pragma unroll
        for (int j = 0; j < 4; ++j) t[j] = Q::clip(div(x[j]), lo, hi);
        w[k] = quant4(t[0], t[1], t[2], t[3]);
    }
}
// the same through the one-operation form: the integer is in the low byte of the clipped sum
template <int DTYPE>
__device__ __forceinline__ void quantize_raw_magic(const uint4 *raw, float r, float lo, float hi, unsigned w[4])
{
    const float mlo = kRoundMagic + lo, mhi = kRoundMagic + hi;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        float x[4];
        unsigned b[4];
        widen4<DTYPE>(raw, k, x);
#pragma unroll
        for (int j = 0; j < 4; ++j) b[j] = __float_as_uint(fmaxf(fminf(__fmaf_rn(x[j], r, kRoundMagic), mhi), mlo));
        w[k] = __byte_perm(__byte_perm(b[0], b[1], 0x0040), __byte_perm(b[2], b[3], 0x0040), 0x5410);
    }
}
// int8 values clipped to four bits at position s (s = 4: any int8), four at a time: with the sign folded away a value
// is out of range where a bit at or above s + 3 is set, and is then replaced by the largest in range
__device__ __forceinline__ unsigned clip_bytes(unsigned w, int s)
{
    const unsigned in_range = (((8u << s) - 1u) & 0x7fu) * 0x01010101u;
    unsigned sign, over;
    asm("prmt.b32 %0, %1, 0, 0xba98;" : "=r"(sign) : "r"(w));
    const unsigned y = w ^ sign;
    asm("prmt.b32 %0, %1, 0, 0xba98;" : "=r"(over) : "r"((y & ~in_range) + 0x7f7f7f7fu));   // 0xff where a byte (at most 0x7f) is not zero
    return ((y | over) & in_range) ^ sign;
}

template <int DTYPE>
__device__ __forceinline__ size_t elem_bytes()
{
    return DTYPE == FLEXIQ_DTYPE_F32 ? 4 : (DTYPE == FLEXIQ_DTYPE_I8 ? 1 : 2);
}

}  // namespace flexiq
