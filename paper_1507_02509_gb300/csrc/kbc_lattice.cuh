// D2Q9 lattice constants and storage codecs for the sm_103a kernels.
//
// Velocity set (Sec. 2): tensor product of {-1, 0, 1}; population index
// i = 3(b+1) + (a+1) for v_i = (a, b).  The weights W_i and cs^2 are not
// printed in the paper (Eq. S, Eq. Eq); the D2Q9 product weights
// W_(a,b) = w_a w_b with w_0 = 2/3, w_{+-1} = 1/6 and cs^2 = 1/3 are used.
//
// Populations are stored as deviations from the rest weights, d_i = f_i - W_i,
// which keeps O(u) information in the leading bits of low-precision storage.
#pragma once

#include <cuda_fp16.h>
#include <cstdint>

namespace kbc {

__host__ __device__ constexpr int va(int i) { return i % 3 - 1; }
__host__ __device__ constexpr int vb(int i) { return i / 3 - 1; }
__host__ __device__ constexpr double w1(int a) { return a == 0 ? 2.0 / 3.0 : 1.0 / 6.0; }
__host__ __device__ constexpr double wgt(int i) { return w1(va(i)) * w1(vb(i)); }
// 1 / W_i: 36 (diagonal), 9 (axis), 9/4 (rest)
__host__ __device__ constexpr double inv_wgt(int i)
{
    return (va(i) != 0 && vb(i) != 0) ? 36.0 : (va(i) == 0 && vb(i) == 0) ? 2.25 : 9.0;
}

template <typename T> __device__ __forceinline__ T fmaT(T a, T b, T c);
template <> __device__ __forceinline__ float fmaT<float>(float a, float b, float c) { return __fmaf_rn(a, b, c); }
template <> __device__ __forceinline__ double fmaT<double>(double a, double b, double c) { return __fma_rn(a, b, c); }

// weight class of population i: 0 diagonal (W = 1/36), 1 axis (1/9), 2 rest (4/9)
__host__ __device__ constexpr int wclass(int i)
{
    return (va(i) != 0 && vb(i) != 0) ? 0 : (va(i) == 0 && vb(i) == 0) ? 2 : 1;
}

// The conversion instructions between 32 and 64 bits take as long as an FP64
// one, also where they are predicated off.  Out of line, so that the branches
// below, which hardly any value takes, stay branches.
static __device__ __noinline__ double cvt_f64(float v) { return (double)v; }
static __device__ __noinline__ float cvt_f32(double v) { return __double2float_rn(v); }

// A float as a double by integer operations; zeros included, subnormal,
// infinite and NaN values by the instruction.
__device__ __forceinline__ double widen(float v)
{
    const unsigned b = __float_as_uint(v), e = (b >> 23) & 0xffu;
    if (e - 1u >= 254u && (b << 1) != 0u) return cvt_f64(v);
    const unsigned m = e == 0u ? 0u : ((b & 0x7fffffffu) >> 3) + 0x38000000u;
    return __hiloint2double((int)(m | (b & 0x80000000u)), (int)(b << 29));
}

// the same for a positive normal float
__device__ __forceinline__ double widen_normal(float v)
{
    const unsigned b = __float_as_uint(v);
    return __hiloint2double((int)((b >> 3) + 0x38000000u), (int)(b << 29));
}

// A double rounded to the nearest float, ties to even: the truncated bits
// plus the rounding, which may carry into the exponent.  Outside the normal
// floats (and for zero) the instruction.
__device__ __forceinline__ float narrow(double v)
{
    const unsigned H = (unsigned)__double2hiint(v), B = (unsigned)__double2loint(v);
    const unsigned e = (H >> 20) & 0x7ffu;
    if (e - 897u >= 254u) return cvt_f32(v);
    const unsigned t = ((e - 896u) << 23) | (__funnelshift_l(B, H, 3) & 0x7fffffu), r = B & 0x1fffffffu;
    const unsigned up = (r + (t & 1u)) > 0x10000000u ? 1u : 0u;
    return __uint_as_float((t + up) | (H & 0x80000000u));
}

// A double rounded to a float whose last bit is set when the value is not
// exact (round to odd), from which rounding on to half gives the nearest half.
__device__ __forceinline__ float narrow_odd(double v)
{
    const unsigned H = (unsigned)__double2hiint(v), B = (unsigned)__double2loint(v);
    const unsigned e = (H >> 20) & 0x7ffu;
    if (e < 897u) return __uint_as_float(H & 0x80000000u);  // a half of zero
    if (e >= 1151u) return cvt_f32(v);
    const unsigned t = ((e - 896u) << 23) | (__funnelshift_l(B, H, 3) & 0x7fffffu);
    return __uint_as_float(t | ((B & 0x1fffffffu) ? 1u : 0u) | (H & 0x80000000u));
}

// The leading 24 bits of a double as a float (truncated), for magnitudes in
// 2^-74 .. 8; 0 below, NaN outside.
__device__ __forceinline__ float leading(double v)
{
    const unsigned H = (unsigned)__double2hiint(v), e = (H >> 20) & 0x7ffu;
    const unsigned f = (__funnelshift_l((unsigned)__double2loint(v), H, 3) & 0x7fffffu) | ((e - 896u) << 23);
    return e < 949u ? 0.0f : e > 1025u ? __uint_as_float(0x7fffffffu) : __uint_as_float(f | (H & 0x80000000u));
}

// out of line for the same reason
static __device__ __noinline__ double divide_one(double x) { return 1.0 / x; }

// 1 / x in double for positive normal x (others by the IEEE division): with
// x = m 2^k, 1 <= m < 2, the single-precision reciprocal y of m's leading bits
// (relative error below 2^-21), then y (1 + r + r^2) with the residual
// r = 1 - m y, whose remainder r^3 is below the last bit: one value in a million
// rounds otherwise than the quotient (30 of 3.4e7, none by more than one unit;
// a refinement of y in single precision made that fewer for random values and
// more, 6.6e4, for those next to powers of two, where the quotients are nearly
// ties).  Three FP64 instructions; the IEEE division takes about nine.
__device__ __forceinline__ double rcp_pos(double x)
{
    const unsigned H = (unsigned)__double2hiint(x), B = (unsigned)__double2loint(x);
    const unsigned e = H >> 20;
    if (e - 1u >= 2044u) return divide_one(x);  // not a positive normal with a normal reciprocal
    const float mf = __uint_as_float(0x3f800000u | (__funnelshift_l(B, H, 3) & 0x7fffffu));
    const double m = __hiloint2double((int)((H & 0xfffffu) | 0x3ff00000u), (int)B);
    const double y = widen_normal(__fdividef(1.0f, mf));
    const double r = __fma_rn(-m, y, 1.0);
    const double z = __fma_rn(y, __fma_rn(r, r, r), y);  // in (1/2, 1]
    return __hiloint2double(__double2hiint(z) + (int)((1023u - e) << 20), __double2loint(z));
}

// Scale of the half-precision encoding (unused by the other codecs): S and,
// per weight class, the decode factor W/S, rounded once on the host so that
// the kernels take it from the parameter bank instead of forming it per
// thread.
struct CodecScale {
    float scale;      // S
    float inv_scale;  // 1 / S
    float dec[3];     // W_c / S
};

__host__ inline CodecScale make_scale(double s)
{
    const double w[3] = {1.0 / 36.0, 1.0 / 9.0, 4.0 / 9.0};
    CodecScale c;
    c.scale = (float)s;
    c.inv_scale = (float)(1.0 / s);
    for (int k = 0; k < 3; ++k) c.dec[k] = (float)(w[k] / s);
    return c;
}

// Storage codecs: S = stored element, T = arithmetic type.
//   decode(s, i, c)     -> d_i = f_i - W_i in T
//   load(s, i, c), store(e, i, c)
//                       -> the step kernels' view: the value the collision
//                          works on, d_i itself, or with kUnits the storage
//                          code in T (the collision's storage units)
//   to_f64(s, i, c)     -> d_i in double (exact for F64/F32 storage)
//   from_f64(d, i, c)   -> stored element from a double deviation
// kVec: nodes per thread of the vector-row kernel (kVec * sizeof(S) bytes
// per load/store; 16 for F64/F32, 8 for F16, which keeps F16 registers low).
// kRowMinBlocks: resident 64-thread blocks per SM the vector-row kernel is
// compiled for.  12 caps it at 80 registers (65536 / (12 * 64) = 85; every
// variant fits without spilling) and keeps 24 warps per SM loading: 3%
// faster than 96 registers for KBC B and 5% for C/D.  Left free,
// the compiler takes up to 190 registers and the bandwidth-bound FP32 step
// loses a third of its rate.  FP64 is bound by its arithmetic pipe, not by
// occupancy.
struct CodecF64 {
    using S = double;
    using T = double;
    static constexpr int kVec = 2;
    static constexpr int kRowMinBlocks = 1;
    static constexpr bool kUnits = false;
    __device__ __forceinline__ static T decode(S s, int, const CodecScale&) { return s; }
    __device__ __forceinline__ static T load(S s, int, const CodecScale&) { return s; }
    __device__ __forceinline__ static S store(T d, int, const CodecScale&) { return d; }
    __device__ __forceinline__ static double to_f64(S s, int, const CodecScale&) { return s; }
    // d_i / W_i in double
    __device__ __forceinline__ static double relative(S s, int i, const CodecScale&) { return s * inv_wgt(i); }
    __device__ __forceinline__ static S from_f64(double d, int, const CodecScale&) { return d; }
};

struct CodecF32 {
    using S = float;
    using T = float;
    static constexpr int kVec = 4;
    static constexpr int kRowMinBlocks = 12;
    static constexpr bool kUnits = false;
    __device__ __forceinline__ static T decode(S s, int, const CodecScale&) { return s; }
    __device__ __forceinline__ static T load(S s, int, const CodecScale&) { return s; }
    __device__ __forceinline__ static S store(T d, int, const CodecScale&) { return d; }
    __device__ __forceinline__ static double to_f64(S s, int, const CodecScale&) { return widen(s); }
    __device__ __forceinline__ static double relative(S s, int i, const CodecScale&) { return widen(s) * inv_wgt(i); }
    __device__ __forceinline__ static S from_f64(double d, int, const CodecScale&) { return narrow(d); }
};

// (f - W)/W * S in IEEE half (stored as its 16-bit pattern), arithmetic in
// float.  The step kernels collide in storage units: load and store are the
// bare conversions.
struct CodecF16 {
    using S = unsigned short;
    using T = float;
    static constexpr int kVec = 4;
    static constexpr int kRowMinBlocks = 12;
    static constexpr bool kUnits = true;
    __device__ __forceinline__ static T load(S s, int, const CodecScale&)
    {
        return __half2float(__ushort_as_half(s));
    }
    __device__ __forceinline__ static S store(T e, int, const CodecScale&)
    {
        return __half_as_ushort(__float2half_rn(e));
    }
    // two populations of the same plane in one packed conversion
    __device__ __forceinline__ static unsigned store2(T e0, T e1, int, const CodecScale&)
    {
        const __half2 h = __floats2half2_rn(e0, e1);
        return *reinterpret_cast<const unsigned*>(&h);
    }
    __device__ __forceinline__ static T decode(S s, int i, const CodecScale& c)
    {
        return __half2float(__ushort_as_half(s)) * c.dec[wclass(i)];
    }
    __device__ __forceinline__ static double to_f64(S s, int i, const CodecScale& c)
    {
        return widen(__half2float(__ushort_as_half(s))) * (wgt(i) * (double)c.inv_scale);
    }
    __device__ __forceinline__ static double relative(S s, int, const CodecScale& c)
    {
        return widen(__half2float(__ushort_as_half(s))) * (double)c.inv_scale;
    }
    __device__ __forceinline__ static S from_f64(double d, int i, const CodecScale& c)
    {
        return __half_as_ushort(__float2half_rn(narrow_odd(d * (inv_wgt(i) * (double)c.scale))));
    }
};

}  // namespace kbc
