// Arithmetic that keeps double-precision results off GB300's FP64 pipe.
//
// An FP64 instruction occupies a quarter of an SM for 64 cycles per warp,
// however many of its lanes are active (measured: 64.1 cycles per DFMA with 1
// to 32 active lanes, one warp per scheduler; conversions between 64-bit and
// 32-bit types 81 to 89), against one cycle for an FP32 or integer
// instruction.  Two tools follow (and rcp_pos in kbc_lattice.cuh, a double
// reciprocal by three fused multiply-adds).
//
// * FF<L>: an unevaluated sum of two floats (Dekker's and Knuth's error-free
//   transformations), 48 bits, in the one-node lane Lf or the packed lane
//   Lf2.  Used where the result is a stored float or half: a bound on the
//   error says whether the rounding to the stored type is settled (Ziv's
//   test); where it is not, the caller computes the node in double.  The
//   stored values are those of the double computation, always.
// * Fixed sums: the nine stored populations as integers in one common unit,
//   exact, so that rho and j are exact integer sums, rounded once.
#pragma once

#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include "kbc_lanes.cuh"
#include "kbc_lattice.cuh"

namespace kbc {

// a - b as one fused operation, also for the packed lane (the product is
// exact, so the rounding is that of the subtraction)
__device__ __forceinline__ Lf subL(Lf a, Lf b) { return a - b; }
__device__ __forceinline__ Lf2 subL(Lf2 a, Lf2 b) { return fmaL(b, Lf2(-1.0f), a); }

template <class L>
struct FF {
    L h, l;
    FF() = default;
    __device__ __forceinline__ FF(L hh, L ll) : h(hh), l(ll) {}
};

// x + y = s + e exactly (Knuth)
template <class L> __device__ __forceinline__ FF<L> two_sum(L x, L y)
{
    const L s = x + y, b = subL(s, x);
    return FF<L>(s, subL(x, subL(s, b)) + subL(y, b));
}
// the same for |x| >= |y| (Dekker)
template <class L> __device__ __forceinline__ FF<L> fast_two_sum(L x, L y)
{
    const L s = x + y;
    return FF<L>(s, subL(y, subL(s, x)));
}
// error <= 2^-47 (|x| + |y|); the second member may exceed half an ulp of
// the first, which every use here allows
template <class L> __device__ __forceinline__ FF<L> add_raw(FF<L> x, FF<L> y)
{
    const FF<L> s = two_sum(x.h, y.h);
    return FF<L>(s.h, s.l + (x.l + y.l));
}
template <class L> __device__ __forceinline__ FF<L> operator+(FF<L> x, FF<L> y)
{
    const FF<L> s = add_raw(x, y);
    return fast_two_sum(s.h, s.l);
}
template <class L> __device__ __forceinline__ FF<L> operator-(FF<L> x) { return FF<L>(-x.h, -x.l); }
template <class L> __device__ __forceinline__ FF<L> operator-(FF<L> x, FF<L> y) { return x + (-y); }
// error <= 2^-45 |x y|
template <class L> __device__ __forceinline__ FF<L> operator*(FF<L> x, FF<L> y)
{
    const L p = x.h * y.h;
    L e = fmaL(x.h, y.h, -p);
    e = fmaL(x.h, y.l, e);
    e = fmaL(x.l, y.h, e);
    return fast_two_sum(p, e);
}
// multiplication by a power of two
template <class L> __device__ __forceinline__ FF<L> scale(FF<L> x, float c) { return FF<L>(x.h * L(c), x.l * L(c)); }

// c rounded to a pair of floats (compile-time constants)
__host__ __device__ constexpr float ff_hi(double c) { return (float)c; }
__host__ __device__ constexpr float ff_lo(double c) { return (float)(c - (double)(float)c); }

// A double as a pair of floats by integer operations (the top 24 bits,
// truncated, and the other 29 rounded to a float): relative error 2^-48.
// Magnitudes below 2^-74 become 0; false from 8 upwards and for NaN.
__device__ __forceinline__ bool split_double(double v, float& h, float& l)
{
    const unsigned H = (unsigned)__double2hiint(v), B = (unsigned)__double2loint(v);
    const unsigned e = (H >> 20) & 0x7ffu, s = H & 0x80000000u;
    h = __uint_as_float(s | ((e - 896u) << 23) | (__funnelshift_l(B, H, 3) & 0x7fffffu));
    l = __uint2float_rn(B & 0x1fffffffu) * __uint_as_float(s | ((e - 948u) << 23));
    if (e < 949u) h = l = 0.0f;
    return e <= 1025u;
}

// The float nearest to s + t, where that is settled for every value within
// err of it (ok is cleared otherwise).
__device__ __forceinline__ void round_sure(float s, float t, float err, float& out, bool& ok)
{
    out = __fadd_rn(s, t);
    ok &= __fadd_rn(s, __fadd_rn(t, -err)) == out && __fadd_rn(s, __fadd_rn(t, err)) == out;
}
// The same for the nearest half.
__device__ __forceinline__ void round_sure(float s, float t, float err, unsigned short& out, bool& ok)
{
    const __half a = __float2half_rn(__fadd_rd(s, __fadd_rd(t, -err)));
    const __half b = __float2half_rn(__fadd_ru(s, __fadd_ru(t, err)));
    out = __half_as_ushort(a);
    if (out != __half_as_ushort(b)) {
        // the two ends of a one-ulp bracket round apart: the halfway value
        // (a float) lies between them
        const float m = 0.5f * (__half2float(a) + __half2float(b));
        const float d = __fadd_rn(__fsub_rn(s, m), t);
        ok &= fabsf(d) > 2.0f * err;
        if (d > 0.0f) out = __half_as_ushort(b);
    }
}

// (1 + x) ln(1 + x) near x = 0 with eight FP64 instructions (the library's
// log1p alone takes about thirty): Taylor's series about the nearest multiple
// m of 1/128, with r = (x - m) / (1 + m),
//   (1 + m) ln(1 + m) + (1 + ln(1 + m)) (x - m)
//     + (x - m) r (1/2 - r/6 + r^2 (1/12 + t)),  t = -r/20 + r^2/30 - r^3/42.
// For |x| < 1/2.  It is no less accurate than (W + d) log1p(d / W): a node's
// entropy has 0.50 to 0.81 times the rms error of that, in a host model over
// relative deviations of 2^-16 to 2^-3, and a mean error below 0.15 of its rms.
// What keeps it there:
// * t in single precision is added to 1/12 as an integer, to 2^-42 (formed in
//   single precision as a whole the bracket was off by up to 2^-43, of one
//   sign: 1.3 times the error near x = 2^-8);
// * the constant terms, which cancel against the linear ones in the sum over a
//   node, are summed as integers in units of 2^-46; what they leave, and what 1
//   + ln(1 + m) in double leaves, enters the series in single precision.
// The table is made at compile time, ln(1 + m) = 2 atanh(j / (256 + j)) for
// m = j / 128 by its series in 100 fractional bits.
struct EntropyTable {
    static constexpr int kHalf = 64, kSize = 2 * kHalf + 1, kUnitBits = 46;
    // 1 + ln(1 + m) and what is left of it; (1 + m) ln(1 + m) in units, and
    // what is left of that
    double m[kSize] = {}, c[kSize] = {}, g[kSize] = {};
    long long units[kSize] = {};
    float g_low[kSize] = {}, f_low[kSize] = {};

    EntropyTable() = default;
    struct Make {};
    __host__ __device__ constexpr explicit EntropyTable(Make)
    {
        using Fixed = __int128;
        constexpr Fixed one = Fixed(1) << 100, unit = one >> kUnitBits;
        for (int k = 0; k < kSize; ++k) {
            const int j = k - kHalf, q = 256 + j;
            Fixed term = j * one / q, log = 0;
            for (int i = 1; i < 80; i += 2) {
                log += 2 * term / i;
                term = term * (j * j) / (q * q);
            }
            m[k] = j / 128.0;
            c[k] = 1.0 / (1.0 + j / 128.0);
            g[k] = double(one + log) * 0x1p-100;
            g_low[k] = float(double(one + log - (long long)(g[k] * 0x1p62) * (one >> 62)) * 0x1p-100);
            const Fixed f = log * (128 + j) / 128;
            units[k] = (long long)((f + (f < 0 ? -unit : unit) / 2) / unit);
            f_low[k] = float(double(f - units[k] * unit) * 0x1p-100);
        }
    }
};
__device__ constexpr EntropyTable kEntropy{EntropyTable::Make()};

// The table in shared memory.
struct EntropyLogs {
    static constexpr int kSize = EntropyTable::kSize;
    double m[kSize], c[kSize], g[kSize];
    long long units[kSize];
    float g_low[kSize], f_low[kSize];
    __device__ __forceinline__ void fill()
    {
        for (int k = threadIdx.x; k < kSize; k += blockDim.x) {
            m[k] = kEntropy.m[k];
            c[k] = kEntropy.c[k];
            g[k] = kEntropy.g[k];
            units[k] = kEntropy.units[k];
            g_low[k] = kEntropy.g_low[k];
            f_low[k] = kEntropy.f_low[k];
        }
    }
    // (1 + x) ln(1 + x) less `unit` units; x in double and as a float (to about 2^-20 of itself)
    __device__ __forceinline__ double near(double x, float xf, long long& unit) const
    {
        const int k = __float2int_rn(xf * (2.0f * EntropyTable::kHalf)) + EntropyTable::kHalf;
        const double d = x - m[k];
        const double r = d * c[k];
        const float mf = (float)(k - EntropyTable::kHalf) * (0.5f / EntropyTable::kHalf), df = xf - mf;
        const float rf = df * __fdividef(1.0f, 1.0f + mf);
        // |t| < 2^-11.3: neither the integer nor the exponent of 1/12 overflows
        const float t = rf * __fmaf_rn(rf, __fmaf_rn(rf, -1.0f / 42.0f, 1.0f / 30.0f), -1.0f / 20.0f);
        const double twelfth = __longlong_as_double(__double_as_longlong(1.0 / 12.0) +
                                                    (long long)__float2int_rn(t * 0x1p42f) * 16384);
        double h = __fma_rn(r, twelfth, -1.0 / 6.0);
        h = __fma_rn(r, h, 0.5);
        unit = units[k];
        return __fma_rn(g[k], d, __fma_rn(d * r, h, widen(__fmaf_rn(g_low[k], df, f_low[k]))));
    }
    // |units| < 2^51 as a double, to be multiplied by 2^-46
    __device__ __forceinline__ static double as_double(long long unit)
    {
        constexpr double two52 = 6755399441055744.0;  // 2^52 + 2^51, whose last bit is 1
        return __longlong_as_double(__double_as_longlong(two52) + unit) - two52;
    }
};

// Exact sums over the nine stored populations as 64-bit integers: with
// the unit double(unit) they are drho = rho - 1, jx and jy.  A value enters
// with its 24 (11) significant bits shifted by its exponent against the
// largest one, at most 30 (29) places, so that no bit is lost and nine
// values stay below 2^59.  False (sums undefined) when a value is not
// finite, a single-precision one is subnormal, or one that is not zero lies more than
// 30 binary places below the largest.
struct FixedSums {
    long long drho, jx, jy;
    double unit;
};

template <class C> struct fixed_of { static constexpr bool kHas = false; };

__device__ __forceinline__ void fixed_combine(const long long (&v)[9], FixedSums& s)
{
    const long long r = v[2] + v[5] + v[8], l = v[0] + v[3] + v[6];
    const long long t = v[6] + v[7] + v[8], b = v[0] + v[1] + v[2];
    s.drho = r + l + (v[1] + v[4] + v[7]);
    s.jx = r - l;
    s.jy = t - b;
}

template <> struct fixed_of<CodecF32> {
    static constexpr bool kHas = true;
    __device__ __forceinline__ static bool sums(const float (&d)[9], const CodecScale&, FixedSums& s)
    {
        unsigned top = 0u;
#pragma unroll
        for (int i = 0; i < 9; ++i) top = max(top, __float_as_uint(d[i]) & 0x7fffffffu);
        const int e = (int)(top >> 23);
        if (e >= 255 || (top != 0u && e < 64)) return false;
        bool ok = true;
        long long v[9];
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            const unsigned b = __float_as_uint(d[i]);
            const int ei = (int)((b >> 23) & 0xffu);
            const int sh = 30 - (e - ei);
            const int m = (int)((b & 0x7fffffu) | 0x800000u);
            const bool zero = (b << 1) == 0u;
            ok &= zero || (sh >= 0 && ei != 0);
            const int sm = zero ? 0 : ((int)b < 0 ? -m : m);
            v[i] = (long long)sm * (long long)(1 << (sh & 31));
        }
        fixed_combine(v, s);
        // unit 2^(e - 127 - 23 - 30)
        s.unit = __hiloint2double((e - 180 + 1023) << 20, 0);
        return ok;
    }
};

template <> struct fixed_of<CodecF16> {
    static constexpr bool kHas = true;
    __device__ __forceinline__ static bool sums(const unsigned short (&c)[9], const CodecScale& cs, FixedSums& s)
    {
        bool ok = true;
        long long v[9];
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            const int ei = (c[i] >> 10) & 31;
            ok &= ei != 31;
            int m = (int)(c[i] & 0x3ffu) | (ei ? 0x400 : 0);
            if (c[i] & 0x8000u) m = -m;
            // times m_i = 36 W_i = 1, 4, 16
            const int sh = (ei ? ei - 1 : 0) + 2 * wclass(i);
            v[i] = (long long)m << sh;
        }
        fixed_combine(v, s);
        // unit W / S 2^-24 of the diagonal populations
        s.unit = (wgt(0) * (double)cs.inv_scale) * 0x1p-24;
        return ok;
    }
};

}  // namespace kbc
