// Device helpers of the GB300 Krylov library: rank lookups, the matrix-free H.v row,
// complex arithmetic and dot-product accumulators.
#pragma once

#include <type_traits>

#include "kry_internal.cuh"

namespace kry {

// ---------------------------------------------------------------- element types

template <class V> struct VT;
template <> struct VT<double2> {
    using R = double;
    __device__ __forceinline__ static double2 zero() { return make_double2(0.0, 0.0); }
    __device__ __forceinline__ static double ehlo(const DevHam &h, uint32_t p) { return __ldg(h.ehlo_d + p); }
    __device__ __forceinline__ static double ehhi(const DevHam &h, uint32_t p) { return __ldg(h.ehhi_d + p); }
    __device__ __forceinline__ static double eh8(const DevHam &h, size_t p) { return __ldg(h.eh8_d + p); }
    __device__ __forceinline__ static double2 from(double2 c) { return c; }
};
template <> struct VT<float2> {
    using R = float;
    __device__ __forceinline__ static float2 zero() { return make_float2(0.f, 0.f); }
    __device__ __forceinline__ static float ehlo(const DevHam &h, uint32_t p) { return __ldg(h.ehlo_f + p); }
    __device__ __forceinline__ static float ehhi(const DevHam &h, uint32_t p) { return __ldg(h.ehhi_f + p); }
    __device__ __forceinline__ static float eh8(const DevHam &h, size_t p) { return __ldg(h.eh8_f + p); }
    __device__ __forceinline__ static float2 from(double2 c) { return make_float2((float)c.x, (float)c.y); }
};

// ---------------------------------------------------------------- float-float vectors
// GB300 runs FP64 arithmetic, and conversions between FP64 and FP32, at 1/64 of its FP32
// rate, so the complex128 passes are bound by the FP64 pipe at about a third of the HBM rate.
// dtype KRY_C128E keeps the Krylov vectors as float-float pairs (ffc, kry_internal.cuh: 16
// bytes per element like complex128, about 48 significant bits) and does all vector
// arithmetic on the FP32 pipe: products are formed exactly for the leading parts (the fused
// multiply-add error term) with the cross terms in float, and sums are float-float (Knuth's
// TwoSum).  A dot product is accurate to about 2^-47 of the sum of |terms| (FP64: 2^-53).
// Complex128 inputs and coefficients are converted at the boundary: a double is split by
// integer operations on its bits into its leading 24 significant bits and the next 23.

__device__ __forceinline__ void ff_combine(float &s, float &c, float s2, float c2);

// hi + lo floats of x (|x| in [2^-80, 2^128); smaller magnitudes give 0, which for vectors of
// norm of order one changes a dot product by less than 2^-80 D^(1/2))
__device__ __forceinline__ float2 dsplit(double x)
{
    const unsigned hw = (unsigned)__double2hiint(x), lw = (unsigned)__double2loint(x);
    const unsigned ex = (hw >> 20) & 0x7ffu;
    const bool ok = ex >= 943u && ex <= 1150u;
    const unsigned sg = hw & 0x80000000u;
    const float hi = __uint_as_float(ok ? (sg | ((ex - 896u) << 23) | ((hw & 0xfffffu) << 3) | (lw >> 29)) : 0u);
    const float lm = __fsub_rn(__uint_as_float(0x4b000000u | ((lw >> 6) & 0x7fffffu)), 8388608.0f);   // exact
    const float sc = __uint_as_float(ok ? (sg | ((ex - 942u) << 23)) : 0u);                            // +-2^(e-46)
    return make_float2(hi, __fmul_rn(lm, sc));
}
// a float as a double, exactly, by integer operations (zero and subnormal floats give 0)
__device__ __forceinline__ double f2d(float f)
{
    const unsigned b = __float_as_uint(f), e = (b >> 23) & 0xffu;
    const unsigned hi = e ? ((b & 0x80000000u) | ((e + 896u) << 20) | ((b & 0x7fffffu) >> 3)) : 0u;
    const unsigned lo = e ? ((b & 7u) << 29) : 0u;
    return __hiloint2double((int)hi, (int)lo);
}
// float-float s + c rounded to FP64 (one FP64 add)
__device__ __forceinline__ double ff2d(float s, float c) { return f2d(s) + f2d(c); }
// (s, c) += (ah + al)(bh + bl): the leading product split exactly (TwoSum into s), the error
// term and the cross terms into c
__device__ __forceinline__ void ff_mac(float ah, float al, float bh, float bl, float &s, float &c)
{
    const float p = __fmul_rn(ah, bh);
    float e = __fmaf_rn(ah, bh, -p);
    e = __fmaf_rn(ah, bl, e);
    e = __fmaf_rn(al, bh, e);
    const float t = __fadd_rn(s, p);
    const float z = __fsub_rn(t, s);
    const float err = __fadd_rn(__fsub_rn(s, __fsub_rn(t, z)), __fsub_rn(p, z));
    s = t;
    c = __fadd_rn(c, __fadd_rn(err, e));
}
// (s, c) renormalised so that |c| is at most half an ulp of s (TwoSum: exact for any order of
// magnitudes, so also after a cancellation has left |c| > |s|)
__device__ __forceinline__ void ff_renorm(float &s, float &c)
{
    const float t = __fadd_rn(s, c);
    const float z = __fsub_rn(t, s);
    c = __fadd_rn(__fsub_rn(s, __fsub_rn(t, z)), __fsub_rn(c, z));
    s = t;
}

template <> struct VT<ffc> {
    using R = double;
    __device__ __forceinline__ static ffc zero() { return ffc{0.f, 0.f, 0.f, 0.f}; }
    __device__ __forceinline__ static double ehlo(const DevHam &h, uint32_t p) { return __ldg(h.ehlo_d + p); }
    __device__ __forceinline__ static double ehhi(const DevHam &h, uint32_t p) { return __ldg(h.ehhi_d + p); }
    __device__ __forceinline__ static double eh8(const DevHam &h, size_t p) { return __ldg(h.eh8_d + p); }
    __device__ __forceinline__ static ffc from(double2 c)
    {
        const float2 a = dsplit(c.x), b = dsplit(c.y);
        return ffc{a.x, b.x, a.y, b.y};
    }
};
__device__ __forceinline__ ffc ldg(const ffc *p)
{
    const float4 v = __ldg((const float4 *)p);
    return ffc{v.x, v.y, v.z, v.w};   // (xh, yh, xl, yl)
}
__device__ __forceinline__ float2 ldg(const float2 *p) { return __ldg(p); }
__device__ __forceinline__ double2 ldg(const double2 *p) { return __ldg(p); }

// *a where p holds, else zero, as one predicated load (a branch around a load costs more than the load)
__device__ __forceinline__ float2 ldg_if(bool p, const float2 *a)
{
    float2 v;
    asm("{.reg .pred q; setp.ne.s32 q, %3, 0; mov.b32 %0, 0; mov.b32 %1, 0; @q ld.global.nc.v2.f32 {%0, %1}, [%2];}"
        : "=&f"(v.x), "=&f"(v.y) : "l"(a), "r"((int)p));
    return v;
}
__device__ __forceinline__ double2 ldg_if(bool p, const double2 *a)
{
    double2 v;
    asm("{.reg .pred q; setp.ne.s32 q, %3, 0; mov.b64 %0, 0; mov.b64 %1, 0; @q ld.global.nc.v2.f64 {%0, %1}, [%2];}"
        : "=&d"(v.x), "=&d"(v.y) : "l"(a), "r"((int)p));
    return v;
}
__device__ __forceinline__ ffc ldg_if(bool p, const ffc *a)
{
    ffc v;
    asm("{.reg .pred q; setp.ne.s32 q, %5, 0; mov.b32 %0, 0; mov.b32 %1, 0; mov.b32 %2, 0; mov.b32 %3, 0; "
        "@q ld.global.nc.v4.f32 {%0, %1, %2, %3}, [%4];}"
        : "=&f"(v.xh), "=&f"(v.yh), "=&f"(v.xl), "=&f"(v.yl) : "l"(a), "r"((int)p));
    return v;
}

// the 16 bytes at p (16-byte aligned): one element, or two of complex64
__device__ __forceinline__ void ldg_chunk(const float2 *p, float2 *dst)
{
    const float4 v = __ldg((const float4 *)p);
    dst[0] = make_float2(v.x, v.y);
    dst[1] = make_float2(v.z, v.w);
}
__device__ __forceinline__ void ldg_chunk(const double2 *p, double2 *dst) { dst[0] = __ldg(p); }
__device__ __forceinline__ void ldg_chunk(const ffc *p, ffc *dst) { dst[0] = ldg(p); }

// Per element type, the accumulator of a neighbour sum: the element itself, or two float-float
// numbers.
struct FF4 {   // two float-float numbers (real, imaginary)
    float sr = 0.f, cr = 0.f, si = 0.f, ci = 0.f;
};
template <class V> struct Arith {
    using HvSum = V;
};
template <> struct Arith<ffc> {
    using HvSum = FF4;
};

__device__ __forceinline__ double2 operator+(double2 a, double2 b) { return make_double2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ float2 operator+(float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); }

// w - c v (complex)
__device__ __forceinline__ double2 cfms(double2 c, double2 v, double2 w)
{
    return make_double2(fma(-c.x, v.x, fma(c.y, v.y, w.x)), fma(-c.x, v.y, fma(-c.y, v.x, w.y)));
}
__device__ __forceinline__ float2 cfms(float2 c, float2 v, float2 w)
{
    return make_float2(fmaf(-c.x, v.x, fmaf(c.y, v.y, w.x)), fmaf(-c.x, v.y, fmaf(-c.y, v.x, w.y)));
}

// d x + s acc  (real d, s)
__device__ __forceinline__ double2 axpby(double d, double2 x, double s, double2 a)
{
    return make_double2(fma(d, x.x, s * a.x), fma(d, x.y, s * a.y));
}
__device__ __forceinline__ float2 axpby(float d, float2 x, float s, float2 a)
{
    return make_float2(fmaf(d, x.x, s * a.x), fmaf(d, x.y, s * a.y));
}
// neighbour sums of the H.v row: acc += v, then y = sd x + shj acc
__device__ __forceinline__ void hv_add(double2 &acc, double2 v) { acc = acc + v; }
__device__ __forceinline__ void hv_add(float2 &acc, float2 v) { acc = __fadd2_rn(acc, v); }
__device__ __forceinline__ void hv_add(FF4 &acc, ffc v)
{
    ff_combine(acc.sr, acc.cr, v.xh, v.xl);
    ff_combine(acc.si, acc.ci, v.yh, v.yl);
}
// acc += v[0] + ... + v[N - 1]
template <int N, class S, class V> __device__ __forceinline__ void hv_add_n(S &acc, const V *v)
{
#pragma unroll
    for (int u = 0; u < N; ++u) hv_add(acc, v[u]);
}
// Neighbour sums of complex128 on 64-bit integers, the real and the imaginary parts each on a scale of their
// own (H is real, so neither part may cost the other accuracy): the mantissas of a part are aligned to its
// largest exponent so far (the sum so far shifted along when it grows), with 5 bits of fraction below and room
// for 32 terms above.  Each term loses less than 2^-56 of the largest of its part (the bits shifted out, and
// one unit for a negative term), an FP64 sum 2^-53 of the running one; a single term is exact.  A term takes
// about 16 integer instructions per part where an FP64 add takes the pipe for 77 issue cycles (L = 24: 213 us
// with FP64 adds, the kernel's bound).
struct ISum {
    long long s = 0;
    unsigned top = 0, low = 0;   // largest high word without its sign, and the low words' bits
    __device__ __forceinline__ static unsigned mag(double x) { return (unsigned)__double2hiint(x) & 0x7fffffffu; }
    // mantissa of x in units of 2^(em - 1080), em >= its exponent; x, or for a negative x its complement.  The
    // shift is clamped to 64 by the instruction.  (A zero or subnormal x counts as 2^-1023 here: from em = 128 on
    // that is shifted out, and below that value() and special() do not use the sum.)
    __device__ __forceinline__ static long long align(double x, unsigned em)
    {
        const unsigned lo = (unsigned)__double2loint(x);
        const unsigned h5 = (__funnelshift_l(lo, (unsigned)__double2hiint(x), 5) & 0x1ffffffu) | 0x2000000u;
        unsigned long long q;
        asm("shr.u64 %0, %1, %2;" : "=l"(q) : "l"((unsigned long long)h5 << 32 | (unsigned long long)(lo << 5)), "r"(em - (mag(x) >> 20)));
        return (long long)q ^ (long long)(__double2hiint(x) >> 31);
    }
    // a and, with PAIR, b
    template <bool PAIR> __device__ __forceinline__ void add(double a, double b)
    {
        const unsigned t = max(top, PAIR ? max(mag(a), mag(b)) : mag(a)), em = t >> 20;
        low |= PAIR ? (unsigned)__double2loint(a) | (unsigned)__double2loint(b) : (unsigned)__double2loint(a);
        asm("shr.s64 %0, %0, %1;" : "+l"(s) : "r"(em - (top >> 20)));
        top = t;
        s += align(a, em);
        if (PAIR) s += align(b, em);
    }
    // infinities, NaN and exponents the scale cannot hold, down to subnormal values: the caller sums the row in
    // FP64
    __device__ __forceinline__ bool special() const
    {
        return top >= 0x7ff00000u || (top < (128u << 20) && (top | low) != 0u);
    }
    __device__ __forceinline__ double value() const
    {
        if (top == 0u) return 0.0;
        return (double)s * __hiloint2double((int)((top >> 20) - 1080u + 1023u) << 20, 0);   // 2^(em - 1075 - 5)
    }
};
struct ISum2 {
    ISum re, im;
    __device__ __forceinline__ bool special() const { return re.special() || im.special(); }
    __device__ __forceinline__ double2 value() const { return make_double2(re.value(), im.value()); }
};
// (two terms at a time whatever N, so that the bits do not depend on how many are loaded together)
template <int N> __device__ __forceinline__ void hv_add_n(ISum2 &acc, const double2 *v)
{
#pragma unroll
    for (int u = 0; u < N; u += 2) {
        acc.re.add<(N > 1)>(v[u].x, v[N > 1 ? u + 1 : u].x);
        acc.im.add<(N > 1)>(v[u].y, v[N > 1 ? u + 1 : u].y);
    }
}
__device__ __forceinline__ void hv_add(ISum2 &acc, double2 v) { hv_add_n<1>(acc, &v); }
template <class V, class R> __device__ __forceinline__ V hv_finish(R sd, V x, R shj, V acc) { return axpby(sd, x, shj, acc); }
__device__ __forceinline__ double2 hv_finish(double sd, double2 x, double shj, const ISum2 &acc)
{
    return axpby(sd, x, shj, acc.value());
}
__device__ __forceinline__ ffc hv_finish(double sd, ffc x, double shj, const FF4 &acc)
{
    const float2 d = dsplit(sd), h = dsplit(shj);
    float sr = 0.f, cr = 0.f, si = 0.f, ci = 0.f;
    ff_mac(d.x, d.y, x.xh, x.xl, sr, cr);
    ff_mac(h.x, h.y, acc.sr, acc.cr, sr, cr);
    ff_mac(d.x, d.y, x.yh, x.yl, si, ci);
    ff_mac(h.x, h.y, acc.si, acc.ci, si, ci);
    ff_renorm(sr, cr);
    ff_renorm(si, ci);
    return ffc{sr, si, cr, ci};
}
__device__ __forceinline__ double2 scale(double2 a, double s) { return make_double2(a.x * s, a.y * s); }
// s a for a float-float element: the product of the split scale with each component
__device__ __forceinline__ ffc scale(ffc a, double s)
{
    const float2 f = dsplit(s);
    float sr = 0.f, cr = 0.f, si = 0.f, ci = 0.f;
    ff_mac(f.x, f.y, a.xh, a.xl, sr, cr);
    ff_mac(f.x, f.y, a.yh, a.yl, si, ci);
    ff_renorm(sr, cr);
    ff_renorm(si, ci);
    return ffc{sr, si, cr, ci};
}
__device__ __forceinline__ float2 scale(float2 a, double s) { return make_float2(a.x * (float)s, a.y * (float)s); }
__device__ __forceinline__ float2 scale(float2 a, float s) { return make_float2(a.x * s, a.y * s); }

// ---------------------------------------------------------------- launch ordering

// First statement of every kernel of the replayed step: wait until the kernel before it
// has completed and its writes are visible (griddepcontrol.wait; it returns at once for a
// kernel launched without programmatic dependence), then let the next kernel begin its
// launch, so that launches overlap the tails of the kernels before them.
__device__ __forceinline__ void pdl_begin()
{
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// ---------------------------------------------------------------- dot accumulators
// sum conj(a) b, complex (the readout <psi0, w>).  complex128: FP64 fused multiply-adds.  complex64 and float-float: every
// product is split exactly (p = a*b rounded, e = fma(a, b, -p)) and summed with Knuth's
// TwoSum into a float pair (s, c): the rounding errors of s are kept exactly, and c gathers
// them in plain float.  c is folded back into s (renorm, a TwoSum) after every few terms --
// the callers do it every few rows -- so that its own rounding stays at 2^-48 of |s|: left to
// grow over the N terms of a thread, c's rounding errors add up to about N 2^-48 of the sum
// (5e-11 relative at N = 16K, the rows per thread of an L = 30 sector).

__device__ __forceinline__ double2 warp_sum(double2 v);

struct DotAccD {
    double re = 0.0, im = 0.0;
    __device__ __forceinline__ void add(double2 a, double2 b)
    {
        re = fma(a.x, b.x, re); re = fma(a.y, b.y, re);
        im = fma(a.x, b.y, im); im = fma(-a.y, b.x, im);
    }
    __device__ __forceinline__ void renorm() {}
    __device__ __forceinline__ double2 value() const { return make_double2(re, im); }
    // the sum over the warp (valid in every lane)
    __device__ __forceinline__ double2 warp_value() const { return warp_sum(value()); }
};

// Float-float sum (s, c) += (s2, c2): TwoSum of the leading parts, the trailing parts and the
// rounding error added, then renormalised.  Symmetric in its two operands.
__device__ __forceinline__ void ff_combine(float &s, float &c, float s2, float c2)
{
    const float t = __fadd_rn(s, s2);
    const float z = __fsub_rn(t, s);
    const float e = __fadd_rn(__fsub_rn(s, __fsub_rn(t, z)), __fsub_rn(s2, z));
    const float cc = __fadd_rn(__fadd_rn(c, c2), e);
    s = __fadd_rn(t, cc);
    c = __fsub_rn(cc, __fsub_rn(s, t));
}
// Sum of a float-float value over the warp, in FP32 arithmetic (GB300 runs FP64, and the
// conversions to it, at 1/64 of the FP32 rate, so per-thread FP64 epilogues of the streaming
// kernels cost as much as their streams at small j): every lane ends with the total.
__device__ __forceinline__ void ff_warp_sum(float &s, float &c)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const float s2 = __shfl_xor_sync(0xffffffffu, s, o), c2 = __shfl_xor_sync(0xffffffffu, c, o);
        ff_combine(s, c, s2, c2);
    }
}

__device__ __forceinline__ void two_sum(float a, float b, float &s, float &e)
{
    s = __fadd_rn(a, b);
    float z = __fsub_rn(s, a);
    e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, z)), __fsub_rn(b, z));
}
__device__ __forceinline__ void exact_fma(float a, float b, float &s, float &c)
{
    float p = __fmul_rn(a, b);
    float e = __fmaf_rn(a, b, -p);
    float t, err;
    two_sum(s, p, t, err);
    s = t;
    c = __fadd_rn(c, __fadd_rn(err, e));
}
struct DotAccF {
    float sr = 0.f, cr = 0.f, si = 0.f, ci = 0.f;
    __device__ __forceinline__ void add(float2 a, float2 b)
    {
        exact_fma(a.x, b.x, sr, cr); exact_fma(a.y, b.y, sr, cr);
        exact_fma(a.x, b.y, si, ci); exact_fma(-a.y, b.x, si, ci);
    }
    __device__ __forceinline__ void renorm()
    {
        ff_renorm(sr, cr);
        ff_renorm(si, ci);
    }
    __device__ __forceinline__ double2 value() const
    {
        return make_double2((double)sr + (double)cr, (double)si + (double)ci);
    }
    __device__ __forceinline__ double2 warp_value() const
    {
        float a = sr, b = cr, c = si, d = ci;
        ff_warp_sum(a, b);
        ff_warp_sum(c, d);
        return make_double2((double)a + (double)b, (double)c + (double)d);
    }
};
// sum conj(a) b for float-float vectors (ffc)
struct DotAccFF {
    float sr = 0.f, cr = 0.f, si = 0.f, ci = 0.f;
    __device__ __forceinline__ void add(ffc a, ffc b)
    {
        ff_mac(a.xh, a.xl, b.xh, b.xl, sr, cr);
        ff_mac(a.yh, a.yl, b.yh, b.yl, sr, cr);
        ff_mac(a.xh, a.xl, b.yh, b.yl, si, ci);
        ff_mac(-a.yh, -a.yl, b.xh, b.xl, si, ci);
    }
    __device__ __forceinline__ void renorm()
    {
        ff_renorm(sr, cr);
        ff_renorm(si, ci);
    }
    __device__ __forceinline__ double2 value() const { return make_double2(ff2d(sr, cr), ff2d(si, ci)); }
    __device__ __forceinline__ double2 warp_value() const
    {
        float a = sr, b = cr, c = si, d = ci;
        ff_warp_sum(a, b);
        ff_warp_sum(c, d);
        return make_double2(ff2d(a, b), ff2d(c, d));
    }
};

template <class V> struct DotAcc;
template <> struct DotAcc<double2> : DotAccD {};
template <> struct DotAcc<float2> : DotAccF {};
template <> struct DotAcc<ffc> : DotAccFF {};

__device__ __forceinline__ double2 warp_sum(double2 v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        v.x += __shfl_xor_sync(0xffffffffu, v.x, o);
        v.y += __shfl_xor_sync(0xffffffffu, v.y, o);
    }
    return v;
}

__device__ __forceinline__ double warp_sum(double v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// ---------------------------------------------------------------- sums without the FP64 pipe
// GB300 issues one FP64 warp instruction per about 77 cycles and SM sub-partition, so the trees and
// gathers that end a reduction cost more in FP64 adds than the loads before them.  These sums align
// the mantissas to the largest exponent of the warp as 64-bit integers, add those exactly (in 26-bit
// limbs, one redux each) and round once: the terms lose less than 2^-54 of the largest each, which
// is no more than the roundings of an FP64 sum of as many, and the order does not matter.

// Integer sum over the warp of CNT values per lane (CNT <= 8): every lane gets S and k with the total
// = S 2^k.  False (uniform) when a value is infinite or NaN, or the largest below 2^-895 and not zero
// (beside larger ones, subnormal values count as zero).
template <int CNT>
__device__ __forceinline__ bool warp_isum(const double *v, long long &S, int &k)
{
    unsigned top = 0;   // largest high word without its sign, not zero for a value that is not
#pragma unroll
    for (int i = 0; i < CNT; ++i)
        top = max(top, ((unsigned)__double2hiint(v[i]) & 0x7fffffffu) | min((unsigned)__double2loint(v[i]), 1u));
    top = __reduce_max_sync(0xffffffffu, top);
    S = 0;
    k = 0;
    if (top == 0u) return true;
    const unsigned em = top >> 20;
    if (em == 0x7ffu || em < 128u) return false;
    constexpr int SH = CNT == 1 ? 5 : 2;   // 53 bits + SH + log2(32 CNT) <= 63
    long long q = 0;
#pragma unroll
    for (int i = 0; i < CNT; ++i) {
        const unsigned hi = (unsigned)__double2hiint(v[i]), lo = (unsigned)__double2loint(v[i]), e = (hi >> 20) & 0x7ffu;
        unsigned long long m = ((unsigned long long)((hi & 0xfffffu) | 0x100000u) << 32 | lo) << SH;
        const unsigned d = em - e;
        m = e == 0u || d > 63u ? 0ull : m >> d;
        q += (int)hi < 0 ? -(long long)m : (long long)m;
    }
    const unsigned mask = (1u << 26) - 1u;
    const unsigned l0 = __reduce_add_sync(0xffffffffu, (unsigned)q & mask);
    const unsigned l1 = __reduce_add_sync(0xffffffffu, (unsigned)(q >> 26) & mask);
    const int l2 = __reduce_add_sync(0xffffffffu, (int)(q >> 52));
    S = (long long)l0 + ((long long)l1 << 26) + ((long long)l2 << 52);
    k = (int)em - 1075 - SH;
    return true;
}
// S 2^k (k >= -1000), rounded once
__device__ __forceinline__ double from_isum(long long S, int k)
{
    return (double)S * __hiloint2double((k + 1023) << 20, 0);
}
// Sum over the warp of CNT values per lane, in every lane.
template <int CNT>
__device__ __forceinline__ double warp_sum_int(const double *v)
{
    long long S;
    int k;
    if (warp_isum<CNT>(v, S, k)) return from_isum(S, k);
    double t = v[0];
#pragma unroll
    for (int i = 1; i < CNT; ++i) t += v[i];
    return warp_sum(t);
}

// ---------------------------------------------------------------- real inner products
// The Hamiltonian is real and symmetric, so the Lanczos process of a complex vector is that of
// H (+) H on its real and imaginary parts: a vector of 2D reals with the inner product
// Re <a, b>.  Its coefficients alpha_j and beta_j are the same, Re <v_i, v_j> = delta_ij is the
// orthogonality it needs, and Im <v_i, v_j> = Im <psi, p_i(H) p_j(H) psi> = 0 by itself, since
// p_i p_j (H) is Hermitian.  Every v_j is a real polynomial of H applied to psi, the Krylov
// approximation of exp(-i tau (H (+) H)) maps to that of exp(-i tau H) by (x, y) -> x + i y,
// and an error of the former grows by at most sqrt(2) under that map.  Full reorthogonalisation
// in this inner product takes half the multiply-adds of the complex one in the dots and in the
// updates, where GB300 is bound by them (FP64 by its 1/64 rate, float-float by its 10 to 12
// instructions per product).  The loss of Re-orthogonality and the errors of psi are those of the
// complex form (tests/test_real_lanczos.py emulates both on the CPU).

struct FF {   // a float-float number
    float s, c;
};
__device__ __forceinline__ FF add2(FF a, FF b)
{
    ff_combine(a.s, a.c, b.s, b.c);
    return a;
}
__device__ __forceinline__ FF shfl_xor(FF v, int o)
{
    return FF{__shfl_xor_sync(0xffffffffu, v.s, o), __shfl_xor_sync(0xffffffffu, v.c, o)};
}
__device__ __forceinline__ FF pick(bool p, FF a, FF b) { return FF{p ? a.s : b.s, p ? a.c : b.c}; }

// Totals over the warp of N values per lane (N a power of two up to 32): lane l returns the total of
// value l / (32 / N).  Doubles as integers; float-float numbers by exchange, N - 1 + log2(32 / N)
// adds per lane instead of 5 N.
template <int N>
__device__ __forceinline__ double warp_totals(double *v)
{
    const int lane = threadIdx.x & 31;
    long long S = 0;
    int k = 0;
    bool ok = true;
#pragma unroll
    for (int i = 0; i < N; ++i) {
        long long Si = 0;
        int ki = 0;
        ok &= warp_isum<1>(v + i, Si, ki);
        if (lane / (32 / N) == i) { S = Si; k = ki; }
    }
    if (ok) return from_isum(S, k);
    double t = 0.0;
#pragma unroll
    for (int i = 0; i < N; ++i) {
        const double w = warp_sum(v[i]);
        if (lane / (32 / N) == i) t = w;
    }
    return t;
}
template <int N, class T>
__device__ __forceinline__ T warp_totals(T *v)
{
    const int lane = threadIdx.x & 31;
    int o = 16;
#pragma unroll
    for (int n = N / 2; n >= 1; n >>= 1, o >>= 1) {
        const bool up = lane & o;
#pragma unroll
        for (int i = 0; i < n; ++i) {
            const T send = pick(up, v[i], v[i + n]), keep = pick(up, v[i + n], v[i]);
            v[i] = add2(keep, shfl_xor(send, o));
        }
    }
#pragma unroll
    for (; o >= 1; o >>= 1) v[0] = add2(v[0], shfl_xor(v[0], o));
    return v[0];
}
__device__ __forceinline__ double add2(double a, double b) { return a + b; }
template <class S> __device__ __forceinline__ S from_double(double v);
template <> __device__ __forceinline__ double from_double<double>(double v) { return v; }
template <> __device__ __forceinline__ FF from_double<FF>(double v)
{
    const float2 f = dsplit(v);
    return FF{f.x, f.y};
}
__device__ __forceinline__ double to_double(double v) { return v; }
__device__ __forceinline__ double to_double(FF v) { return (double)v.s + (double)v.c; }

// Accumulators of sum Re(conj(a) b), with b prepared once for several vectors (Pre).
// complex128: two FP64 multiply-adds per element.
template <class V> struct RealAcc;
template <> struct RealAcc<double2> {
    using Pre = double2;
    using Sum = double;
    double s = 0.0;
    __device__ __forceinline__ static Pre pre(double2 b) { return b; }
    __device__ __forceinline__ void add(double2 a, Pre b) { s = fma(a.x, b.x, s); s = fma(a.y, b.y, s); }
    __device__ __forceinline__ void renorm() {}
    __device__ __forceinline__ Sum sum() const { return s; }
};
__device__ __forceinline__ float2 fsub2(float2 a, float2 b) { return __ffma2_rn(b, make_float2(-1.f, -1.f), a); }
__device__ __forceinline__ float2 neg2(float2 a) { return make_float2(-a.x, -a.y); }
// s + c += -n + e with n = -(a product rounded) and e its exact remainder: TwoSum into s, the
// errors into c, two float-float lanes per packed FP32x2 instruction
__device__ __forceinline__ void ff2_add_neg(float2 &s, float2 &c, float2 n, float2 e)
{
    const float2 t = fsub2(s, n);
    const float2 z = fsub2(t, s);
    const float2 err = fsub2(fsub2(s, fsub2(t, z)), __fadd2_rn(n, z));
    s = t;
    c = __fadd2_rn(c, __fadd2_rn(err, e));
}
// (s, c) renormalised by TwoSum, two float-float lanes per instruction
__device__ __forceinline__ void ff_renorm2(float2 &s, float2 &c)
{
    const float2 t = __fadd2_rn(s, c);
    const float2 z = fsub2(t, s);
    c = __fadd2_rn(fsub2(s, fsub2(t, z)), fsub2(c, z));
    s = t;
}
// complex64 and float-float: the lanes of a packed pair sum the products of the real and of the
// imaginary parts, error-free products and TwoSum as in DotAccF; Pre keeps -b too, so that no
// instruction is spent on a sign.
struct RealAccPair {
    using Sum = FF;
    float2 s = make_float2(0.f, 0.f), c = make_float2(0.f, 0.f);
    __device__ __forceinline__ void renorm() { ff_renorm2(s, c); }
    __device__ __forceinline__ Sum sum() const { return add2(FF{s.x, c.x}, FF{s.y, c.y}); }
};
template <> struct RealAcc<float2> : RealAccPair {
    using Pre = float4;   // (b, -b)
    __device__ __forceinline__ static Pre pre(float2 b) { return make_float4(b.x, b.y, -b.x, -b.y); }
    __device__ __forceinline__ void add(float2 a, const Pre &b)
    {
        const float2 n = __fmul2_rn(a, make_float2(b.z, b.w));
        ff2_add_neg(s, c, n, __ffma2_rn(a, make_float2(b.x, b.y), n));
    }
};
struct FFPre {
    float2 h, l, n;   // hi, lo, -hi
};
template <> struct RealAcc<ffc> : RealAccPair {
    using Pre = FFPre;
    __device__ __forceinline__ static Pre pre(ffc b)
    {
        return FFPre{make_float2(b.xh, b.yh), make_float2(b.xl, b.yl), make_float2(-b.xh, -b.yh)};
    }
    __device__ __forceinline__ void add(ffc a, const Pre &b)
    {
        const float2 h = make_float2(a.xh, a.yh), l = make_float2(a.xl, a.yl);
        const float2 n = __fmul2_rn(h, b.n);
        float2 e = __ffma2_rn(h, b.h, n);
        e = __ffma2_rn(h, b.l, e);
        e = __ffma2_rn(l, b.h, e);
        ff2_add_neg(s, c, n, e);
    }
};

// Linear combinations with real coefficients: w -= c x, with -c kept (RCoef).
template <class V> struct RealLin;
template <> struct RealLin<double2> {
    using RCoef = double;
    double2 w;
    __device__ __forceinline__ static RCoef coef(double c) { return -c; }
    RealLin() = default;
    __device__ __forceinline__ RealLin(double2 src) : w(src) {}
    __device__ __forceinline__ void fms(RCoef nc, double2 x) { w.x = fma(nc, x.x, w.x); w.y = fma(nc, x.y, w.y); }
    __device__ __forceinline__ void add(double2 p) { w.x += p.x; w.y += p.y; }
    __device__ __forceinline__ double2 out() const { return w; }
};
template <> struct RealLin<float2> {
    using RCoef = float;
    float2 w;
    __device__ __forceinline__ static RCoef coef(double c) { return -(float)c; }
    RealLin() = default;
    __device__ __forceinline__ RealLin(float2 src) : w(src) {}
    __device__ __forceinline__ void fms(RCoef nc, float2 x) { w = __ffma2_rn(make_float2(nc, nc), x, w); }
    __device__ __forceinline__ void add(float2 p) { w = __fadd2_rn(w, p); }
    __device__ __forceinline__ float2 out() const { return w; }
};
template <> struct RealLin<ffc> {
    using RCoef = float2;   // -c as hi, lo
    float2 s, c;
    __device__ __forceinline__ static RCoef coef(double v)
    {
        const float2 a = dsplit(v);
        return neg2(a);
    }
    RealLin() = default;
    __device__ __forceinline__ RealLin(ffc src) : s(make_float2(src.xh, src.yh)), c(make_float2(src.xl, src.yl)) {}
    __device__ __forceinline__ void fms(RCoef nc, ffc x)
    {
        const float2 h = make_float2(x.xh, x.yh), l = make_float2(x.xl, x.yl);
        const float2 n = __fmul2_rn(make_float2(-nc.x, -nc.x), h);
        float2 e = __ffma2_rn(make_float2(nc.x, nc.x), h, n);
        e = __ffma2_rn(make_float2(nc.x, nc.x), l, e);
        e = __ffma2_rn(make_float2(nc.y, nc.y), h, e);
        ff2_add_neg(s, c, n, e);
    }
    __device__ __forceinline__ void add(ffc p)
    {
        ff2_add_neg(s, c, make_float2(-p.xh, -p.yh), make_float2(p.xl, p.yl));
    }
    __device__ __forceinline__ ffc out()
    {
        ff_renorm2(s, c);
        return ffc{s.x, s.y, c.x, c.y};
    }
};

// The update's terms i < j - 1.  In exact arithmetic only c_j and c_{j-1} differ from zero; the others
// are the rounding of the process (about 2^-50 ||u|| in complex128, 2^-45 in float-float) and the
// subtraction of their multiples keeps the basis orthogonal.  Where sum_{i<j-1} c_i^2 <=
// (ETA ||u||)^2 they are summed in FP32 and taken off w once: FP32 loses 2^-23 of each term, so
// at most 2^-23 sqrt(30) ETA ||u|| in all, 2^-60 (complex128) or 2^-56 (float-float) of ||u||, below
// the rounding of w itself (2^-53, 2^-48); larger coefficients take the full arithmetic.  This moves
// all but two of the j + 1 terms off the FP64 pipe (two cycles of it per SM, 77 per warp, a
// multiply-add) and off the 12-instruction float-float products.  Scales 2^-40 <= sigma_i <= 2^40 keep
// the elements and coefficients inside the FP32 range.
template <class V> struct MinorSum {
    static constexpr bool use = false;   // complex64: the full arithmetic is FP32 already
    static constexpr double eta = 0.0;
};
template <> struct MinorSum<double2> {
    static constexpr bool use = true;
    static constexpr double eta = 9.094947017729282e-13;   // 2^-40
    // the leading 24 bits of a double (|x| < 2^128; below 2^-126 gives 0), by integer operations: the
    // conversion instruction runs at the FP64 rate
    __device__ __forceinline__ static float lead(double x)
    {
        const int hi = __double2hiint(x), v = (hi & 0x7fffffff) - 0x38000000;
        const unsigned b = __funnelshift_l((unsigned)__double2loint(x), (unsigned)v, 3);
        return __uint_as_float((v > 0 ? b : 0u) | ((unsigned)hi & 0x80000000u));
    }
    __device__ __forceinline__ static float2 lead(double2 x) { return make_float2(lead(x.x), lead(x.y)); }
    __device__ __forceinline__ static void add(RealLin<double2> &l, float2 f) { l.w.x += f2d(f.x); l.w.y += f2d(f.y); }
};
template <> struct MinorSum<ffc> {
    static constexpr bool use = true;
    static constexpr double eta = 1.4551915228366852e-11;   // 2^-36
    __device__ __forceinline__ static float2 lead(ffc x) { return make_float2(x.xh, x.yh); }
    __device__ __forceinline__ static void add(RealLin<ffc> &l, float2 f) { l.c = __fadd2_rn(l.c, f); }
};

// Linear combinations with complex coefficients (the combine psi = beta V y): w -= c x.
template <class V> struct CplxLin {
    using RCoef = V;
    V w;
    __device__ __forceinline__ static RCoef coef(double2 c) { return VT<V>::from(c); }
    CplxLin() = default;
    __device__ __forceinline__ CplxLin(V src) : w(src) {}
    __device__ __forceinline__ void fms(RCoef c, V x) { w = cfms(c, x, w); }
    __device__ __forceinline__ V out() const { return w; }
};
template <> struct CplxLin<ffc> {
    using RCoef = float4;   // -(re hi, re lo, im hi, im lo)
    RealLin<ffc> w;
    __device__ __forceinline__ static RCoef coef(double2 c)
    {
        const float2 a = dsplit(c.x), b = dsplit(c.y);
        return make_float4(-a.x, -a.y, -b.x, -b.y);
    }
    CplxLin() = default;
    __device__ __forceinline__ CplxLin(ffc src) : w(src) {}
    // re -= cr xr - ci xi, im -= cr xi + ci xr: a real multiple of x, then one of i x
    __device__ __forceinline__ void fms(RCoef c, ffc x)
    {
        w.fms(make_float2(c.x, c.y), x);
        w.fms(make_float2(c.z, c.w), ffc{-x.yh, x.xh, -x.yl, x.xl});
    }
    __device__ __forceinline__ ffc out() { return w.out(); }
};

// ---------------------------------------------------------------- reductions over the CTAs

// Write this CTA's partials, then let the last CTA to finish sum all partials into
// fin[0..PSTRIDE).  Returns true in the last CTA (all its threads).  Only the slots [0, nlead)
// and, with tail set, SLOT_NRM and SLOT_G are summed (the others of fin are zero): a warp takes a
// slot, lane l the partials of CTAs l, l + 32, ..., eight loads at a time.  With cplx unset the imaginary parts are zero and not summed.  The order depends only on the grid,
// the block and the slot count, so results are bitwise reproducible.
__device__ __forceinline__ bool finish_partials(const double2 *red, double2 *part, KryCtl *ctl,
                                                double2 *fin, int *flag, unsigned *counter = nullptr,
                                                int nlead = PSTRIDE, bool tail = true, bool cplx = true)
{
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nw = blockDim.x >> 5;
    if (!counter) counter = &ctl->counter;
    if (tid < PSTRIDE) part[(size_t)blockIdx.x * PSTRIDE + tid] = red[tid];
    __syncthreads();
    if (tid == 0) {   // (one fence for the CTA: the barrier orders the others' writes before it)
        __threadfence();
        *flag = (atomicAdd(counter, 1u) == gridDim.x - 1) ? 1 : 0;
        __threadfence();
    }
    __syncthreads();
    if (!*flag) return false;
    // slots 0 .. nlead - 1, then NRM and G unless they are among those
    const int nt = tail ? (nlead <= SLOT_NRM ? 2 : 0) : 0, ns = nlead + nt;
    if (tid < PSTRIDE) fin[tid] = make_double2(0.0, 0.0);
    __syncthreads();
    for (int q = warp; q < ns; q += nw) {
        const int slot = q < nlead ? q : SLOT_NRM + (q - nlead);
        if (!cplx && slot == SLOT_G) continue;
        double2 sum = make_double2(0.0, 0.0);
        for (unsigned c0 = 0; c0 < gridDim.x; c0 += 256) {
            double x[8], y[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const unsigned c = c0 + 32 * i + lane;
                double2 v = make_double2(0.0, 0.0);
                if (c < gridDim.x) v = __ldcg(part + (size_t)c * PSTRIDE + slot);
                x[i] = v.x;
                y[i] = v.y;
            }
            sum.x += warp_sum_int<8>(x);
            if (cplx) sum.y += warp_sum_int<8>(y);
        }
        if (lane == 0) fin[slot] = sum;
    }
    __syncthreads();
    return true;
}

// beta_j = ||w|| and the scale of the next vector, or the end of the Krylov space
__device__ __forceinline__ void finalize_beta(KryCtl *ctl, int jj, double nw2, double2 gdot)
{
    const double bt = sqrt(nw2);
    ctl->beta[jj] = bt;
    if (!(nw2 > ctl->eta_bd * ctl->eta_bd * ctl->normu2)) {   // invariant subspace (or zero vector)
        ctl->m_eff = jj + 1;
        ctl->n_bd += 1;
    } else {
        const double s = 1.0 / bt;
        ctl->sigma[jj + 1] = s;
        ctl->g[jj + 1] = make_double2(gdot.x * s, gdot.y * s);
    }
}

// ---------------------------------------------------------------- the H.v's end in the one-read form

// alpha_j = sigma_j Re <W_j, u> from the threads' sums, and in the last CTA the update's coefficients (see
// k_ortho).  The terms C_ki d_k are at the level of the dots d, so FP32 holds them: it loses 2^-24 of each.
// Both are free of H's scale (C_ki is kept over beta_i), so that FP32 holds them for any of it.
// In the first Krylov step v_0 = psi0 / ||psi0||, and P = |sum_i <psi0, v_i> y_i|^2 sees every other vector's
// component along it at first order.  There c_0 is the dot with the u that was stored, whose rounding the
// recurrence does not know, so that the update takes that off along psi0 as well: a basis state's is u's
// element r0, a general state's the sum a0 (A0).  (With c_0 from the recurrence the rounding of u[r0] stayed in
// W_2, W_3, ...: L = 20, N = 7 c64, P at t = 0.05 off by 5.5e-10 instead of 7e-13.)
__device__ __forceinline__ double real_part(const float2 *p) { return (double)__ldcg(p).x; }
__device__ __forceinline__ double real_part(const double2 *p) { return __ldcg(p).x; }
__device__ __forceinline__ double real_part(const ffc *p)
{
    const float4 v = __ldcg((const float4 *)p);
    return (double)v.x + (double)v.z;
}
// first: c_0 is taken here (not the first index of the first step).
template <class V, bool A0>
__device__ __forceinline__ void alpha_epilogue(RealAcc<V> &al, RealAcc<V> &a0, bool first, const V *U, double2 *part,
                                               KryCtl *ctl, int jj)
{
    __shared__ double2 red[PSTRIDE];
    __shared__ double wsum[1 + A0][32];
    __shared__ float Cs[MMAX * MMAX], ds[MMAX + 1];
    __shared__ int flag;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, r0 = ctl->r0;
    const int ns = A0 && first ? 2 : 1;
    al.renorm();
    typename RealAcc<V>::Sum v[1] = {al.sum()};
    const double t = to_double(warp_totals<1>(v));
    if (lane == 0) wsum[0][warp] = t;
    if (A0 && first) {
        a0.renorm();
        typename RealAcc<V>::Sum v0[1] = {a0.sum()};
        const double t0 = to_double(warp_totals<1>(v0));
        if (lane == 0) wsum[A0][warp] = t0;
    }
    if (tid < PSTRIDE) red[tid] = make_double2(0.0, 0.0);
    __syncthreads();
    if (tid < ns) {
        double s = 0.0;
        for (int w = 0; w < (int)blockDim.x / 32; ++w) s += wsum[tid][w];
        red[tid].x = s;
    }
    __syncthreads();
    if (!finish_partials(red, part, ctl, red, &flag, nullptr, ns, false, false)) return;
    double c0 = 0.0;
    if (first && lane == 0) c0 = A0 ? red[A0].x : real_part(U + r0);
    for (int e = tid; e < MMAX * MMAX; e += blockDim.x) Cs[e] = ctl->C[e / MMAX][e % MMAX];
    if (tid <= MMAX) ds[tid] = tid < jj ? ctl->d[tid] : 0.f;   // (d_j = 1 stands apart)
    __syncthreads();
    if (tid >= 64) return;   // lane i for vector i; warp 1 tests the sizes (MinorSum)
    const bool inv = lane <= jj;
    const double s = inv ? ctl->sigma[lane] : 0.0, alpha = red[0].x * ctl->sigma[jj];
    double c = 0.0;
    if (lane < jj) {
        float f = 0.f;
        for (int k = 0; k <= lane; ++k) f = fmaf(Cs[k * MMAX + lane], ds[k], f);
        const double b = ctl->beta[lane];
        const bool sub = lane == jj - 1;   // d_j = 1
        c = fma(b, (double)(sub ? f : f + ds[lane + 1]), sub ? b : 0.0);
    } else if (lane == jj) {
        c = alpha;
    }
    if (first && lane == 0) c = s * c0;
    const double cc = c * c;
    if (warp == 1) {
        bool minor = false;
        if (MinorSum<V>::use) {
            // rounding level, against ||u||^2 >= alpha_j^2 + beta_{j-1}^2
            const bool small = lane + 1 < jj;
            const double cm = small ? cc : 0.0, m2 = warp_sum_int<1>(&cm), big = small ? 0.0 : cc, b2 = warp_sum_int<1>(&big);
            minor = __all_sync(0xffffffffu, !small || (s >= 0x1p-40 && s <= 0x1p40)) &&
                    m2 <= MinorSum<V>::eta * MinorSum<V>::eta * b2;
        }
        if (lane == 0) ctl->minor = minor ? 1 : 0;
        return;
    }
    if (inv) ctl->coefA[lane] = c * s;
    const double c2 = warp_sum_int<1>(&cc);
    if (lane != 0) return;
    ctl->alpha[jj] = alpha;
    ctl->c2 = c2;
    ctl->n_hv += 1;
    ctl->vec_passes += 2;
    ctl->vp_kind[KIND_HV] += 2;   // the H.v: v_j read, u written
    ctl->counter = 0;
}

__device__ __forceinline__ void prefetch_l2(const void *p) { asm volatile("prefetch.global.L2 [%0];" ::"l"(p)); }

// ---------------------------------------------------------------- the one-read pass: rows
// (k_ortho, k_ortho_b)

// Threads of a CTA (one per SM): 16 vectors' rows and accumulators take 96 to 128 registers.
template <class V> constexpr int ORTHO_NTHR = std::is_same<V, ffc>::value ? 384 : 512;
constexpr int ORTHO_QV = 16;   // vectors of a group, at most
constexpr int ORTHO_XU = 2;    // units of a team between two barriers, at most

// The loop is instantiated for 1, 2, 3, 4, 6, 8, 10, 12, 14, 15 and 16 vectors: empty slots of a group of n.
__device__ __forceinline__ int ortho_pad(int n) { return n <= 4 || n == 15 ? 0 : n & 1; }

// What a group of T threads does besides its own vectors' terms and dots: FIRST stores w and takes ||w||^2
// and <psi0, w>, LAST holds u and the terms j - 1 and j.
enum { ORTHO_FIRST = 1, ORTHO_LAST = 2, ORTHO_ONLY = 3 };

// The row loop for one of the CTA's NG groups: the nq = NQ or NQ - 1 vectors from i0 on (the first of NQ slots is empty in
// the latter case), NU units of `unit` elements at a time (thread t of the group takes element t of a unit).
// The vectors' elements are read once, kept in registers, and used for the update and for the dots with its
// result; with two groups to a team their partial updates meet in shared memory (two buffers, one barrier
// per NU units).  The coefficient of vector i is coef[i * cs], its FP32 form mcoef[i * cs].
// A group waits for its loads, then computes, and 16 vectors' rows leave no registers for the next ones: the
// next units' lines are brought into L2 meanwhile (P at L = 24 c64 72.3 -> 69.7 ms, c128 63.1 -> 61.4, L = 30
// c64 247 -> 237, L = 20 with K = 64 88.1 -> 80.7).
template <class V, int NQ, int NU, int KIND, int T, int NG, int B>
__device__ __forceinline__ void ortho_rows(const V *W, size_t ldW, const V *U, const V *G, V *out, size_t n, uint32_t unit,
                                           uint32_t t, int i0, int nq, bool minor, int rp, uint32_t first, uint32_t du,
                                           uint32_t nu, bool back, const typename RealLin<V>::RCoef *coef,
                                           const float *mcoef, int cs, V *xch, RealAcc<V> *acc, RealAcc<V> &nrm,
                                           DotAcc<V> &gacc)
{
    // (single realisations index rows by 32 bits, batched ones elements of [D][K] by 64)
    using idx_t = typename std::conditional<B == 1, uint32_t, size_t>::type;
    constexpr uint32_t FOLD = 8;   // elements between two foldings of the float-float compensations
    constexpr bool LAST = KIND & ORTHO_LAST, FIRST = KIND & ORTHO_FIRST;
    constexpr int NMAJ = NQ < 2 ? 1 : 2;   // (LAST) terms j - 1 and j
    const int pad = NQ - nq;
    const V *Wg = W + (ptrdiff_t)(i0 - pad) * (ptrdiff_t)ldW;   // (slot 0 is not read where pad is 1)
    const int step = B == 1 ? 1 : cs;
    coef += i0 * step;
    mcoef += i0 * step;
    uint32_t it = 0;
    for (uint32_t u0 = first; u0 < nu; u0 += NU * du) {
        {   // the next units' lines into L2, one line per thread of the group
            constexpr int LPU = T * (int)sizeof(V) / 128, NL = NQ * NU * LPU;
#pragma unroll
            for (int e0 = 0; e0 < NL; e0 += T) {
                const int e = e0 + (int)t, q = e / (NU * LPU), line = e % LPU;
                const uint32_t u = u0 + (NU + e / LPU % NU) * du;
                if ((NL % T == 0 || e < NL) && q >= pad && u < nu) {
                    const idx_t rr = (idx_t)(back ? nu - 1 - u : u) * unit + line * (128 / (int)sizeof(V));
                    if (rr < (idx_t)n) prefetch_l2(Wg + (size_t)q * ldW + rr);
                }
            }
        }
        idx_t r[NU];
        V x[NU][NQ], uu[NU];
#pragma unroll
        for (int k = 0; k < NU; ++k) {
            const uint32_t u = u0 + k * du;
            r[k] = u < nu && t < unit ? (idx_t)(back ? nu - 1 - u : u) * unit + t : (idx_t)n;
            const bool in = r[k] < (idx_t)n;
            uu[k] = VT<V>::zero();
            if (LAST) uu[k] = ldg_if(in, U + r[k]);
            x[k][0] = ldg_if(in && pad == 0, Wg + r[k]);
#pragma unroll
            for (int q = 1; q < NQ; ++q) x[k][q] = ldg_if(in, Wg + (size_t)q * ldW + r[k]);
        }
        // this group's share of w = u - sum c_i W_i; terms at rounding level in FP32
        RealLin<V> l[NU];
        float2 f[NU];
#pragma unroll
        for (int k = 0; k < NU; ++k) {
            l[k] = RealLin<V>(uu[k]);
            f[k] = make_float2(0.f, 0.f);
        }
        if (MinorSum<V>::use && minor) {
            if constexpr (MinorSum<V>::use) {
#pragma unroll
                for (int q = 0; q < NQ; ++q) {
                    const int i = (q == 0 ? 0 : q - pad) * step;   // (an empty slot's x is zero)
#pragma unroll
                    for (int k = 0; k < NU; ++k) {
                        if (LAST && q >= NQ - NMAJ) l[k].fms(coef[i], x[k][q]);
                        else f[k] = __ffma2_rn(make_float2(mcoef[i], mcoef[i]), MinorSum<V>::lead(x[k][q]), f[k]);
                    }
                }
#pragma unroll
                for (int k = 0; k < NU; ++k)
                    if (LAST) MinorSum<V>::add(l[k], f[k]);
            }
        } else {
#pragma unroll
            for (int q = 0; q < NQ; ++q)
#pragma unroll
                for (int k = 0; k < NU; ++k) l[k].fms(coef[(q == 0 ? 0 : q - pad) * step], x[k][q]);
        }
        if (KIND != ORTHO_ONLY) {
            // publish this share, meet, take the team's other one: w = LAST's + FIRST's
            V *buf = xch + ((it & 1) * NG + 2 * rp) * T * ORTHO_XU + t;
#pragma unroll
            for (int k = 0; k < NU; ++k) {
                if (LAST) buf[T * k] = l[k].out();
                else if (MinorSum<V>::use && minor) *(float2 *)(buf + T * (ORTHO_XU + k)) = f[k];
                else buf[T * (ORTHO_XU + k)] = l[k].out();
            }
            asm volatile("bar.sync %0, %1;" ::"r"(1 + rp), "n"(2 * T) : "memory");
#pragma unroll
            for (int k = 0; k < NU; ++k) {
                if (!LAST) l[k] = RealLin<V>(buf[T * k]);
                if (MinorSum<V>::use && minor) {
                    if constexpr (MinorSum<V>::use)
                        MinorSum<V>::add(l[k], LAST ? *(const float2 *)(buf + T * (ORTHO_XU + k)) : f[k]);
                } else {
                    l[k].add(buf[T * (ORTHO_XU + k)]);
                }
            }
        }
#pragma unroll
        for (int k = 0; k < NU; ++k) {
            if (NU > 1 && KIND == ORTHO_ONLY && u0 + k * du >= nu) break;
            const V w = l[k].out();
            const typename RealAcc<V>::Pre p = RealAcc<V>::pre(w);
            if (FIRST) nrm.add(w, p);
#pragma unroll
            for (int q = 0; q < NQ; ++q) acc[q].add(x[k][q], p);
            if (FIRST && r[k] < (idx_t)n) {
                out[r[k]] = w;
                if (G) gacc.add(ldg(G + r[k]), w);
            }
        }
        it += 1;
        if (it % (FOLD / NU) == 0) {
#pragma unroll
            for (int q = 0; q < NQ; ++q) acc[q].renorm();
            nrm.renorm();
            gacc.renorm();
        }
    }
}

// ---------------------------------------------------------------- rank tables

// Locate rank r0 + t (< D) as (block hi, offset in block, particles in the lower part):
// start from the block of the enclosing tile's first rank and step over whole blocks.
__device__ __forceinline__ void tile_unrank(const DevBasis &b, const uint32_t *bsz_s, uint32_t r0,
                                            uint32_t t, uint32_t &hi, uint32_t &off, int &klo)
{
    const uint32_t nhi = 1u << b.Lhi;
    uint32_t h = __ldg(b.tstart + r0 / (uint32_t)TILE);
    uint32_t o = r0 - __ldg(b.blk + h) + t;
    int k = b.N - __popc(h);
    while (o >= bsz_s[k]) {
        o -= bsz_s[k];
        do { ++h; k = b.N - __popc(h); } while ((k < 0 || k > b.Llo) && h + 1 < nhi);
        if (k < 0 || k > b.Llo) { k = 0; o = 0; break; }   // unreachable when r0 + t < D
    }
    hi = h; off = o; klo = k;
}

// Stage the small tables (and optionally ranklo, 2^Llo 16-bit entries) in shared memory.
__device__ __forceinline__ void stage_tables(const DevBasis &b, uint32_t *koff_s, uint32_t *bsz_s,
                                             uint16_t *rl_s, int rl_smem)
{
    for (int i = threadIdx.x; i < b.Llo + 2; i += blockDim.x) koff_s[i] = __ldg(b.koff + i);
    for (int i = threadIdx.x; i < b.Llo + 1; i += blockDim.x) bsz_s[i] = __ldg(b.bsz + i);
    if (rl_smem) {
        const uint32_t n2 = (1u << b.Llo) >> 1;   // Llo >= 1, so the count is even
        const uint32_t *src = (const uint32_t *)b.ranklo;
        uint32_t *dst = (uint32_t *)rl_s;
        for (uint32_t i = threadIdx.x; i < n2; i += blockDim.x) dst[i] = __ldg(src + i);
    }
}

// ---------------------------------------------------------------- matrix-free H.v
// Row r of sigma H x for the state s = (hi << Llo) | lo (Eq. 1, XXZ form):
//   (H x)[r] = d(s) x[r] + (J/2) sum_{antiparallel bonds b} x[rank(s ^ bondmask_b)],
//   d(s) = (J Delta / 4)(nbonds - 2 n_anti(s)) + sum_i h_i (n_i - 1/2),
// with sigma folded into the two factors and the bond energy read from a table dz[n_anti].
// Pull form, one writer per row, no atomics.  Rows of upper parts hi with the same particle number
// have the same list of lower parts, so a warp takes an item: 32 consecutive lower parts (one per
// lane) of NH such blocks.  What depends on lo alone -- the ranks of its hops, rl[lo ^ (3 << p)] --
// is found once per item and serves NH rows; what depends on hi alone -- the block starts of its hops
// -- is found once per item by one lane per (block, bond) and shared.  A row then needs no unranking: about 350
// thread instructions in all at L = 24 (c64, 13 hops, alpha_j included; every lower bond is issued for all lanes,
// with or without a hop), 40 us without alpha_j, 138 at L = 26.
// A per-row form (unrank, then a loop over the row's hops) took 404 instructions per row at L = 24
// and 533 at L = 28 without alpha_j, was bound by their issue (59% active) and took 51 us (L = 24 c64).
// The terms of a row are added in bond order, the ring bond last.
constexpr int HV_NH = 8;        // blocks of an item, at most
constexpr int HV_NTHR = 256;    // threads of a CTA of the H.v

// Items by the particle number c of the upper part (its lower part has N - c).
struct HvPlan {
    uint32_t first[18];   // first item of class c
    uint32_t hoff[18];    // first entry of class c in hilist
    uint32_t nlo[17];     // lower parts of class c
    uint32_t koff[17];    // their first position in lolist
    int nh;               // blocks per item
};
struct HvWarp {   // shared memory of a warp
    int steps[HV_NH][24];   // per block: block-start steps of its antiparallel upper bonds (at most 15), packed
    uint32_t hi[HV_NH], base[HV_NH], cross[HV_NH], ring[HV_NH];
    int n[HV_NH];
    uint16_t lower[16][32];   // per lane: ranks of its lower part's hops, packed (complex128 with ALPHA)
};

// With ALPHA *al also sums Re <x, y> over the rows.
template <class V, int RND, int URND, bool ALPHA>
__device__ __forceinline__ void hv_items(const DevBasis &b, const DevHam &hm, const HvPlan &pl, const V *__restrict__ x,
                                         V *__restrict__ y, HvWarp &w, const typename VT<V>::R *dz,
                                         typename VT<V>::R sigma, typename VT<V>::R sigma_halfJ, RealAcc<V> *al)
{
    using R = typename VT<V>::R;
    const int Llo = b.Llo, Lhi = b.Lhi, nlb = Llo - 1, lane = threadIdx.x & 31;
    const uint32_t total = pl.first[Lhi + 1], nw = blockDim.x >> 5;
    int c = 0;
    for (uint32_t item = blockIdx.x * nw + (threadIdx.x >> 5); item < total; item += gridDim.x * nw) {
        while (item >= pl.first[c + 1]) ++c;
        const uint32_t nlo = pl.nlo[c], nch = (nlo + 31u) >> 5, rem = item - pl.first[c], g = rem / nch;
        const uint32_t i = (rem - g * nch) * 32u + lane;   // this lane's lower part
        const uint32_t h0 = pl.hoff[c] + g * pl.nh;
        const int nh = min((uint32_t)pl.nh, pl.hoff[c + 1] - h0);
        // lower part
        const bool valid = i < nlo;
        const uint32_t pos = pl.koff[c] + (valid ? i : 0u), lo = __ldg(b.lolist + pos);
        // upper parts: half a warp per block, lane q for bond q
        __syncwarp();
        for (int j = 0; j < nh; j += 2) {
            const int hh = j + (lane >> 4), q = lane & 15;
            const bool on = hh < nh;
            const uint32_t hi = on ? __ldg(b.hilist + h0 + hh) : 0u;
            const bool aq = on && q < Lhi - 1 && (((hi ^ (hi >> 1)) >> q) & 1u);
            const uint32_t base = __ldg(b.blk + hi);
            const uint32_t to = aq ? __ldg(b.blk + (hi ^ (3u << q))) : 0u;
            const unsigned am = (__ballot_sync(0xffffffffu, aq) >> (lane & 16)) & 0xffffu;
            if (aq) w.steps[hh][__popc(am & ((1u << q) - 1u))] = (int)(to - base);
            if (on && q == 0) {
                w.hi[hh] = hi;
                w.base[hh] = base;
                w.n[hh] = __popc(am);
            }
            if (on && q == 1 && Lhi > 0) w.cross[hh] = __ldg(b.blk + (hi ^ 1u));
            if (on && q == 2 && Lhi > 0) w.ring[hh] = __ldg(b.blk + (hi ^ (1u << (Lhi - 1))));
        }
        const R eh = VT<V>::ehlo(hm, pos);
        const uint32_t anti = valid ? (lo ^ (lo >> 1)) & ((1u << nlb) - 1u) : 0u;
        const uint32_t lomask = (1u << Llo) - 1u;
        // Ranks of the lower part's hops (any pattern has one), in registers; for complex128 with ALPHA packed
        // per lane in shared memory: the rows' loops then run to the longest list of the warp (about nine hops
        // at L = 24) instead of over all Llo - 1 bonds, and its sum costs 32 instructions a term (189 -> 163
        // us).  The other types lose what it takes to pack (L = 26 c64 138 -> 153 us).
        constexpr bool PACK = ALPHA && std::is_same<V, double2>::value;
        uint32_t t[16];
        const int cnt = __popc(anti), most = PACK ? __reduce_max_sync(0xffffffffu, cnt) : nlb;
#pragma unroll
        for (int p0 = 0; p0 < 16; p0 += 4) {
            if (p0 < nlb) {
#pragma unroll
                for (int u = 0; u < 4; ++u) t[p0 + u] = __ldg(b.ranklo + ((lo ^ (3u << (p0 + u))) & lomask));
            }
        }
        if (PACK) {
#pragma unroll
            for (int p = 0; p < 16; ++p)
                if ((anti >> p) & 1u) w.lower[__popc(anti & ((1u << p) - 1u))][lane] = (uint16_t)t[p];
        }
        const uint32_t tc = __ldg(b.ranklo + (lo ^ (1u << nlb))), tr = __ldg(b.ranklo + (lo ^ 1u));
        __syncwarp();
#pragma unroll 1
        for (int h = 0; h < nh; ++h) {
            const uint32_t hi = w.hi[h], base = w.base[h];
            const int n = w.n[h];
            const V *xb = x + base, *xr = xb + i;
            const bool pc = valid && Lhi > 0 && (((lo >> nlb) ^ hi) & 1u);                         // joining bond
            const bool pr = valid && hm.pbc && Lhi > 0 && (((hi >> (Lhi - 1)) ^ lo) & 1u);         // ring bond
            const V x0 = ldg_if(valid, xr);
            auto neighbours = [&](auto &acc) {
                const V vc = ldg_if(pc, x + w.cross[h] + tc), vr = ldg_if(pr, x + w.ring[h] + tr);
                if (PACK) {
#pragma unroll 1
                    for (int k0 = 0; k0 < most; k0 += RND) {   // (entries past a lane's own are not used)
                        V v[RND];
#pragma unroll
                        for (int u = 0; u < RND; ++u) v[u] = ldg_if(k0 + u < cnt, xb + w.lower[(k0 + u) & 15][lane]);
                        hv_add_n<RND>(acc, v);
                    }
                } else {
#pragma unroll
                    for (int p0 = 0; p0 < 16; p0 += RND) {
                        if (p0 < nlb) {
                            V v[RND];
#pragma unroll
                            for (int u = 0; u < RND; ++u) v[u] = ldg_if(anti & (1u << (p0 + u)), xb + t[p0 + u]);
                            hv_add_n<RND>(acc, v);
                        }
                    }
                }
                hv_add(acc, vc);
#pragma unroll 1
                for (int i0 = 0; i0 < n; i0 += URND) {
                    V v[URND];
#pragma unroll
                    for (int u = 0; u < URND; ++u) {   // (entries past n are not used)
                        const bool on = valid && (u == 0 || i0 + u < n);
                        v[u] = ldg_if(on, xr + w.steps[h][i0 + u]);
                    }
                    hv_add_n<URND>(acc, v);
                }
                hv_add(acc, vr);
            };
            const R d = dz[__popc(anti) + n + (int)pc + (int)pr] + eh + VT<V>::ehhi(hm, hi);
            V out;
            if constexpr (std::is_same<V, double2>::value) {   // on aligned integers, in FP64 where they cannot
                ISum2 acc{};
                neighbours(acc);
                if (acc.special()) {   // (a row's own decision: its bits do not depend on the warp's other rows)
                    double2 a2 = VT<V>::zero();
                    neighbours(a2);
                    out = hv_finish(sigma * d, x0, sigma_halfJ, a2);
                } else {
                    out = hv_finish(sigma * d, x0, sigma_halfJ, acc);
                }
            } else {
                typename Arith<V>::HvSum acc{};
                neighbours(acc);
                out = hv_finish(sigma * d, x0, sigma_halfJ, acc);
            }
            if (valid) y[base + i] = out;
            if (ALPHA) al->add(x0, RealAcc<V>::pre(valid ? out : VT<V>::zero()));
        }
        if (ALPHA) al->renorm();   // (once per item, at most eight rows)
    }
}

// *acc sums Re <x, y> over the rows that this thread has written in hv_items.  (A pass of its own: in
// hv_items' loop its accumulators and loads cost every step 2%, c128e at L = 23, for what the first one needs.)
template <class V>
__device__ __forceinline__ void hv_items_dot(const DevBasis &b, const HvPlan &pl, const V *__restrict__ x, const V *y,
                                             RealAcc<V> *acc)
{
    const int lane = threadIdx.x & 31;
    const uint32_t total = pl.first[b.Lhi + 1], nw = blockDim.x >> 5;
    int c = 0;
    for (uint32_t item = blockIdx.x * nw + (threadIdx.x >> 5); item < total; item += gridDim.x * nw) {
        while (item >= pl.first[c + 1]) ++c;
        const uint32_t nlo = pl.nlo[c], nch = (nlo + 31u) >> 5, rem = item - pl.first[c], g = rem / nch;
        const uint32_t i = (rem - g * nch) * 32u + lane, h0 = pl.hoff[c] + g * pl.nh;
        const int nh = min((uint32_t)pl.nh, pl.hoff[c + 1] - h0);
        if (i < nlo) {
            for (int h = 0; h < nh; ++h) {
                const uint32_t r = __ldg(b.blk + __ldg(b.hilist + h0 + h)) + i;
                acc->add(ldg(x + r), RealAcc<V>::pre(y[r]));
            }
        }
        acc->renorm();
    }
}

}  // namespace kry
