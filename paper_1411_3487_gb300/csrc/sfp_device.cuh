// sfp_device.cuh -- device helpers shared by the kernels of the GB300 path:
// the counter-based noise generator and the per-bead normals.
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

namespace sfp {

// Philox4x32-10 (Salmon, Moraes, Dror, Shaw, SC'11): ten rounds of two
// 32x32->64-bit multiplies with a Weyl-sequence key schedule.  Counter
// (step_lo, step_hi, index, tag), key (seed, job_id).
__device__ __forceinline__ uint4 philox4x32_10(uint4 c, uint2 k)
{
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        if (r) { k.x += 0x9E3779B9u; k.y += 0xBB67AE85u; }
        // each multiply as one 32 x 32 -> 64-bit product (both halves at once)
        const uint64_t p0 = (uint64_t)0xD2511F53u * c.x, p1 = (uint64_t)0xCD9E8D57u * c.z;
        const uint32_t lo0 = (uint32_t)p0, hi0 = (uint32_t)(p0 >> 32);
        const uint32_t lo1 = (uint32_t)p1, hi1 = (uint32_t)(p1 >> 32);
        c = make_uint4(hi1 ^ c.y ^ k.x, lo1, hi0 ^ c.w ^ k.y, lo0);
    }
    return c;
}

// Open-interval uniform from the top 23 bits: exact in FP32 (u01_2 below) and
// FP64, so the FP32 and FP64 paths see bit-identical uniforms.
__device__ __forceinline__ double u01d(uint32_t x)
{
    return (double)(x >> 9) * 1.1920928955078125e-07 + 5.9604644775390625e-08;
}

// Pairs of FP32 values in one 64-bit register (fma.rn.f32x2 and relatives: two
// operations, each rounded as on its own, in one instruction).
typedef unsigned long long f32x2;
__device__ __forceinline__ f32x2 pack2(float a, float b)
{
    f32x2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ void unpack2(f32x2 x, float& a, float& b) { asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(x)); }
__device__ __forceinline__ f32x2 both2(float a) { return pack2(a, a); }
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c)
{
    f32x2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b)
{
    f32x2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b)
{
    f32x2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f32x2 sub2(f32x2 a, f32x2 b) { return fma2(b, both2(-1.0f), a); }   // one rounding, as a - b
__device__ __forceinline__ float sqrt_approx(float x)
{
    float r;
    asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// The uniforms (k + 1/2) 2^-23 of two words from their mantissa bits: 1 + k 2^-23
// minus 1 - 2^-24, exact.
__device__ __forceinline__ f32x2 u01_2(uint32_t x, uint32_t y)
{
    return add2(pack2(__uint_as_float((x >> 9) | 0x3f800000u), __uint_as_float((y >> 9) | 0x3f800000u)), both2(-0.99999994f));
}

// FP32 Box-Muller for two word pairs at once (Box and Muller, Ann. Math. Stat. 29
// (1958) 610).  The normals are most of a step's arithmetic, so logarithm, sine and
// cosine are minimax polynomials over the ranges that uniforms of 23 bits can
// reach (coefficients by Remez exchange: no special cases, two arguments per
// instruction): 103 instructions per Philox call of four normals, 178 with logf,
// sincospif and rsqrtf; 96 calls on 16 warps of an SM take 2.16 us, 2.93 us before.
// Over 4 M calls the normals are 4.65e-8 (rms, relative) and 2.1e-7 (largest) off the
// FP64 ones, 5.5e-8 and 2.6e-7 before.
//
// sqrt(-2 ln u): u = 2^e m with m in [sqrt(1/2), sqrt(2)), -2 ln u = -2 e ln 2 +
// f P(f), f = m - 1 (relative error of f P below 2.7e-8).
__device__ __forceinline__ void box_radius2(uint32_t x, uint32_t y, float& ra, float& rb)
{
    float u0, u1;
    unpack2(u01_2(x, y), u0, u1);
    const int i0 = (__float_as_int(u0) - 0x3f3504f3) & (int)0xff800000, i1 = (__float_as_int(u1) - 0x3f3504f3) & (int)0xff800000;
    const f32x2 f = add2(pack2(__int_as_float(__float_as_int(u0) - i0), __int_as_float(__float_as_int(u1) - i1)), both2(-1.0f));
    f32x2 p = both2(-1.744471937e-01f);
    p = fma2(p, f, both2(2.873369157e-01f));
    p = fma2(p, f, both2(-2.990453243e-01f));
    p = fma2(p, f, both2(3.312478662e-01f));
    p = fma2(p, f, both2(-3.991366625e-01f));
    p = fma2(p, f, both2(5.000414848e-01f));
    p = fma2(p, f, both2(-6.666837335e-01f));
    p = fma2(p, f, both2(9.999997616e-01f));
    p = fma2(p, f, both2(-2.0f));
    float a, b;
    unpack2(fma2(p, f, mul2(pack2((float)i0, (float)i1), both2(-1.652591718e-07f))), a, b);   // -2 ln 2 / 2^23 per exponent unit
    ra = sqrt_approx(a);
    rb = sqrt_approx(b);
}

// sin and cos of 2 pi u: 4 u = q + t with q the nearest integer, t in [-1/2, 1/2];
// sin(pi/2 t) and cos(pi/2 t) as polynomials (errors below 4e-9 and 1e-10), swapped
// and signed by the quadrant q.
__device__ __forceinline__ void box_angle2(uint32_t x, uint32_t y, float& s0, float& c0, float& s1, float& c1)
{
    const f32x2 u = u01_2(x, y);
    const f32x2 w = fma2(u, both2(4.0f), both2(12582912.0f));        // 1.5 2^23 + q
    const f32x2 t = fma2(u, both2(4.0f), sub2(both2(12582912.0f), w));
    const f32x2 z = mul2(t, t);
    f32x2 p = fma2(both2(-4.601657856e-03f), z, both2(7.968003303e-02f));
    p = fma2(p, z, both2(-6.459634900e-01f));
    p = fma2(p, z, both2(-4.371139e-08f));                            // pi/2 - fl(pi/2)
    const f32x2 S = fma2(t, both2(1.57079637f), mul2(t, p));
    f32x2 C = fma2(both2(9.033621172e-04f), z, both2(-2.085993625e-02f));
    C = fma2(C, z, both2(2.536691725e-01f));
    C = fma2(C, z, both2(-1.233700514f));
    C = fma2(C, z, both2(1.0f));
    float w0, w1, a0, a1, b0, b1;
    unpack2(w, w0, w1);
    unpack2(S, a0, a1);
    unpack2(C, b0, b1);
    const uint32_t q0 = __float_as_uint(w0), q1 = __float_as_uint(w1);
    s0 = __uint_as_float(__float_as_uint(q0 & 1u ? b0 : a0) ^ ((q0 << 30) & 0x80000000u));
    c0 = __uint_as_float(__float_as_uint(q0 & 1u ? a0 : b0) ^ (((q0 + 1u) << 30) & 0x80000000u));
    s1 = __uint_as_float(__float_as_uint(q1 & 1u ? b1 : a1) ^ ((q1 << 30) & 0x80000000u));
    c1 = __uint_as_float(__float_as_uint(q1 & 1u ? a1 : b1) ^ (((q1 + 1u) << 30) & 0x80000000u));
}

// Bead noise (Eq. b5).  The normals of one chain and step are numbered
// k = 3 n + alpha (bead n, axis alpha); normal k is value k % 4 of Philox call
// k / 4, counter (step_lo, step_hi, call, tag), key (seed, job).  A call gives
// four normals by Box-Muller on its word pairs (0,1) and (2,3), both values of
// each pair used.  Beads 4t .. 4t+3 (12 normals) take exactly calls 3t .. 3t+2.
template <typename T> struct Normals;
template <> struct Normals<float> {
    static __device__ __forceinline__ void draw4(uint32_t seed, uint32_t job, int64_t step,
                                                 uint32_t call, uint32_t tag, float g[4])
    {
        const uint4 w = philox4x32_10(
            make_uint4((uint32_t)step, (uint32_t)((uint64_t)step >> 32), call, tag), make_uint2(seed, job));
        float ra, rb, sa, ca, sb, cb;
        box_radius2(w.x, w.z, ra, rb);
        box_angle2(w.y, w.w, sa, ca, sb, cb);
        // rounded here: a product contracted into a caller's sum would differ between kernels
        g[0] = __fmul_rn(ra, ca); g[1] = __fmul_rn(ra, sa); g[2] = __fmul_rn(rb, cb); g[3] = __fmul_rn(rb, sb);
    }
};
template <> struct Normals<double> {
    static __device__ __forceinline__ void draw4(uint32_t seed, uint32_t job, int64_t step,
                                                 uint32_t call, uint32_t tag, double g[4])
    {
        const uint4 w = philox4x32_10(
            make_uint4((uint32_t)step, (uint32_t)((uint64_t)step >> 32), call, tag), make_uint2(seed, job));
        const double ra = sqrt(-2.0 * log(u01d(w.x)));
        const double rb = sqrt(-2.0 * log(u01d(w.z)));
        double sa, ca, sb, cb;
        sincospi(2.0 * u01d(w.y), &sa, &ca);
        sincospi(2.0 * u01d(w.w), &sb, &cb);
        g[0] = ra * ca; g[1] = ra * sa; g[2] = rb * cb; g[3] = rb * sb;
    }
};

// The normals of beads 4t .. 4t+3 of one chain and step: z[alpha][i] is bead
// 4t + i, axis alpha (calls 3t, 3t+1, 3t+2).
template <typename T>
__device__ __forceinline__ void bead_quad_normals(uint32_t seed, uint32_t job, int64_t step, uint32_t t,
                                                  uint32_t tag, T z[3][4])
{
    T g[3][4];
#pragma unroll
    for (int c = 0; c < 3; ++c) Normals<T>::draw4(seed, job, step, 3u * t + (uint32_t)c, tag, g[c]);
#pragma unroll
    for (int k = 0; k < 12; ++k) z[k % 3][k / 3] = g[k / 4][k % 4];
}

template <typename T> __device__ __forceinline__ T rsqrt_t(T x);
template <> __device__ __forceinline__ float rsqrt_t<float>(float x) { return rsqrtf(x); }
// FP64: the FP32 approximation y (22 bits) and one cubic step, y + y e (1/2 + 3/8 e) with
// e = 1 - x y^2 (the binomial series of (1 - e)^(-1/2), its next term below 2^-63): five
// FP64 instructions, conversions by the bits.  Out of the range of an FP32 seed, and for
// zeros, infinities and NaN, CUDA's own.
template <> __device__ __forceinline__ double rsqrt_t<double>(double x)
{
    const int hi = __double2hiint(x);
    if ((unsigned)(hi - 0x3C300000) >= 0x07800000u) return rsqrt(x);       // 2^-60 <= x < 2^60
    float f = __uint_as_float(((unsigned)(hi - 0x38000000) << 3) | ((unsigned)__double2loint(x) >> 29));
    asm("rsqrt.approx.ftz.f32 %0, %0;" : "+f"(f));
    const unsigned b = __float_as_uint(f);
    const double y = __hiloint2double((int)((b >> 3) + 0x38000000u), (int)(b << 29));
    const double e = fma(-(x * y), y, 1.0);
    return fma(y * e, fma(0.375, e, 0.5), y);
}

}  // namespace sfp
