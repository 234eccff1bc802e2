// exact64.cuh -- correctly rounded IEEE double operations on the integer and
// FP32 pipes.
//
// GB300 issues two FP64 operations per clock and SM, so one FP64 warp
// instruction holds that pipe for 16 cycles, in which the SM's four schedulers
// can issue 64 instructions on its other pipes; a correctly rounded square
// root or division takes about nine such operations. The EXACT64 kernels are
// bound by that pipe, so the operations below leave it: each gives the same
// 64 bits as the IEEE operation it replaces (round to nearest even), for every
// operand in its stated range, and the callers send the others (subnormal,
// infinite, NaN, a result out of the normal range) to the FP64 instruction.
//
// Square root and quotient: a float estimate from the hardware reciprocal
// square root, one Newton correction in float (about 43 bits), the exact
// residual of those bits in 64-bit integers (only its low 64 bits are formed:
// it is known to be small), a second correction from it (within 2^-9 of a
// unit in the last place), and then the final rounding decided exactly by the
// sign of an integer residual: the candidate R of sqrt(X) is the nearest
// integer iff -R < X - R^2 <= R, and C of N/R iff |2 (N - C R)| < R (a quotient
// of two 53-bit significands is never half way between two of them, nor is a
// square root, so no tie arises). Products: the 106-bit integer product of
// the significands, rounded with its round and sticky bits.
//
// Measured (EXACT64, one time step, by events on 16-row tiles): 2048^2 composite on
// the tile kernel 1,267 -> 488 us (169 -> 49 FP64 warp instructions per 32 particles;
// 481 on 8-row tiles, tile2d.cu; single launches under ncu 1,492 -> 476), 1000 x 700
// 236 -> 93 us, the 90 x 81 x 77 foam on the spring lists 151 -> 70 us (30 -> 6
// per 32 springs). What stays on the FP64 pipe: the vector's subtractions, the
// sum of the squares, r - r0, the gather and the integration.
//
// The file also compiles as host code (the estimate is then the caller's), so
// that the arithmetic is tested on the CPU against the C operators.
#pragma once

#include <stdint.h>

#ifdef __CUDACC__
#define LSM_HD __host__ __device__ __forceinline__
#else
#include <cmath>
#include <cstring>
#define LSM_HD inline
#endif

namespace lsm {

LSM_HD uint64_t e64_bits(double d)
{
#ifdef __CUDA_ARCH__
    return (uint64_t)__double_as_longlong(d);
#else
    uint64_t u;
    memcpy(&u, &d, 8);
    return u;
#endif
}

LSM_HD double e64_double(uint64_t u)
{
#ifdef __CUDA_ARCH__
    return __longlong_as_double((long long)u);
#else
    double d;
    memcpy(&d, &u, 8);
    return d;
#endif
}

LSM_HD float e64_f(uint32_t u)
{
#ifdef __CUDA_ARCH__
    return __uint_as_float(u);
#else
    float f;
    memcpy(&f, &u, 4);
    return f;
#endif
}

LSM_HD uint32_t e64_u(float f)
{
#ifdef __CUDA_ARCH__
    return __float_as_uint(f);
#else
    uint32_t u;
    memcpy(&u, &f, 4);
    return u;
#endif
}

LSM_HD float e64_fma(float a, float b, float c)
{
#ifdef __CUDA_ARCH__
    return __fmaf_rn(a, b, c);
#else
    return std::fmaf(a, b, c);
#endif
}

LSM_HD float e64_fmul(float a, float b)
{
#ifdef __CUDA_ARCH__
    return __fmul_rn(a, b);
#else
    return a * b;
#endif
}

LSM_HD uint64_t e64_mulhi(uint64_t a, uint64_t b)
{
#ifdef __CUDA_ARCH__
    return __umul64hi(a, b);
#else
    return (uint64_t)(((unsigned __int128)a * b) >> 64);
#endif
}

// Biased exponent, and the 53-bit significand of a normal double.
LSM_HD int e64_exp(uint64_t u) { return (int)(u >> 52) & 0x7FF; }
LSM_HD uint64_t e64_sig(uint64_t u) { return (u & 0xFFFFFFFFFFFFFull) | 0x10000000000000ull; }

// Whether a double is +0 or -0. On its 32-bit halves: the compiler turns a test
// of the whole word into an FP64 comparison with 0.0 (measured: 8 of the 14
// FP64 instructions that the 3D spring pass had left).
LSM_HD bool e64_zero(uint64_t u) { return ((((uint32_t)(u >> 32)) << 1) | (uint32_t)u) == 0u; }

// The nearest integer to f, |f| < 2^22: f + 1.5 2^23 has it in its low bits.
constexpr float E64_MAGIC = 12582912.0f;
LSM_HD int e64_magic(float f_plus_magic) { return (int)(e64_u(f_plus_magic) - 0x4B400000u); }

// m 2^(x - 52) (m a 53-bit significand, x 0 or 1) as two floats, hi its top
// 24 bits, lo the other 29 bits to float precision.
LSM_HD void e64_split(uint64_t m, unsigned x, float &hi, float &lo)
{
    hi = e64_f(((127u + x) << 23) | ((uint32_t)(m >> 29) & 0x7FFFFFu));
    lo = e64_fmul((float)(int)((uint32_t)m & 0x1FFFFFFFu), e64_f((127u - 52u + x) << 23));
}

// f in [1, 2] in units of 2^-23 (f clamped to that range).
LSM_HD uint32_t e64_fix23(float f) { return e64_u(f) - 0x3F800000u + 0x800000u; }
LSM_HD float e64_clamp12(float f) { return f < 1.0f ? 1.0f : (f > 2.0f ? 2.0f : f); }

// Square root of a positive normal double, and what a division by it needs.
struct Root64 {
    uint64_t R;  // significand
    int e;       // biased exponent
    float y;     // 1 / (R 2^-52) to about 2^-22.9
};

// The argument of the float estimate: x scaled by an even power of two into [1, 4).
LSM_HD float e64_sqrt_arg(uint64_t x)
{
    const unsigned odd = ((unsigned)e64_exp(x) & 1u) ^ 1u;
    return e64_f(((127u + odd) << 23) | ((uint32_t)(x >> 29) & 0x7FFFFFu));
}

// x: bits of a positive normal double; y: 1 / sqrt(e64_sqrt_arg(x)) within
// 2^-22 relative.
LSM_HD Root64 e64_sqrt(uint64_t x, float y)
{
    const int e = e64_exp(x);
    const unsigned odd = ((unsigned)e & 1u) ^ 1u;
    const uint64_t m = e64_sig(x);
    float mh, ml;
    e64_split(m, odd, mh, ml);
    const float g0 = e64_clamp12(e64_fmul(mh, y));
    const float rho = e64_fma(-g0, g0, mh) + ml;
    // about 43 bits of the root, in units of 2^-42
    const uint64_t G = ((uint64_t)e64_fix23(g0) << 19) +
                       (uint64_t)(int64_t)e64_magic(e64_fma(rho, e64_fmul(y, 0x1p41f), E64_MAGIC));
    const int64_t E = (int64_t)((m << (32 + odd)) - G * G);  // (M - G^2) 2^84, below 2^46
    const int D = e64_magic(e64_fma((float)(int)(E >> 16), e64_fmul(y, 0x1p-17f), E64_MAGIC));
    uint64_t R = (G << 10) + (uint64_t)(int64_t)D;            // in units of 2^-52, within one unit
    const int64_t ER = (int64_t)((m << (52 + odd)) - R * R);  // (M - R^2) 2^104
    if (ER > (int64_t)R) R += 1;
    else if (ER <= -(int64_t)R) R -= 1;
    Root64 r;
    r.R = R;
    r.e = (e + 1023) >> 1;
    r.y = y;
    return r;
}

LSM_HD double e64_root(const Root64 &r) { return e64_double(((uint64_t)(r.e - 1) << 52) + r.R); }

// Whether e64_div covers a / r: a normal and the quotient well inside the
// normal range (r normal).
LSM_HD bool e64_div_ok(uint64_t a, const Root64 &r)
{
    const int ea = e64_exp(a);
    return ea >= 1 && ea <= 2046 && (unsigned)(ea - r.e + 1020) < 2040u;
}

// a / r for the bits of a normal double a (e64_div_ok).
LSM_HD double e64_div(uint64_t a, const Root64 &r)
{
    const uint64_t K0 = e64_sig(a);
    const unsigned sh = K0 < r.R ? 1u : 0u;  // the quotient's significand in [1, 2)
    const uint64_t K = K0 << sh;
    float kh, kl, rh, rl;
    e64_split(K0, sh, kh, kl);
    e64_split(r.R, 0u, rh, rl);
    const float q0 = e64_clamp12(e64_fmul(kh, r.y));
    const float rem = e64_fma(-q0, rl, e64_fma(-q0, rh, kh)) + kl;
    const uint64_t Q = ((uint64_t)e64_fix23(q0) << 19) +
                       (uint64_t)(int64_t)e64_magic(e64_fma(rem, e64_fmul(r.y, 0x1p42f), E64_MAGIC));
    const int64_t E = (int64_t)((K << 42) - Q * r.R);  // (K - Q R) 2^94, below 2^54
    const int D = e64_magic(e64_fma((float)(int)(E >> 23), e64_fmul(r.y, 0x1p-19f), E64_MAGIC));
    uint64_t C = (Q << 10) + (uint64_t)(int64_t)D;
    const int64_t EC = (int64_t)((K << 52) - C * r.R) * 2;
    if (EC > (int64_t)r.R) C += 1;
    else if (EC < -(int64_t)r.R) C -= 1;
    const int eq = e64_exp(a) - r.e + 1023 - (int)sh;
    return e64_double((a & 0x8000000000000000ull) | (((uint64_t)(eq - 1) << 52) + C));
}

// Whether e64_prod covers a b: both normal, the product well inside the
// normal range.
LSM_HD bool e64_prod_ok(uint64_t a, uint64_t b)
{
    const int ea = e64_exp(a), eb = e64_exp(b);
    return (unsigned)(ea - 1) < 2046u && (unsigned)(eb - 1) < 2046u && (unsigned)(ea + eb - 1028) < 2036u;
}

// a b for the bits of two normal doubles (e64_prod_ok).
LSM_HD double e64_prod(uint64_t a, uint64_t b)
{
    const uint64_t A = e64_sig(a) << 11, B = e64_sig(b) << 1;
    uint64_t hi = e64_mulhi(A, B), lo = A * B;  // significand product 2^12: hi in [2^52, 2^54)
    const unsigned n = (unsigned)(hi >> 53);
    if (n) {
        lo = (lo >> 1) | (lo & 1) | (hi << 63);
        hi >>= 1;
    }
    // round to nearest even: the fraction lo / 2^64 against one half
    const uint64_t up = (lo >> 63) & (uint64_t)(((lo << 1) != 0) | (hi & 1));
    const int e = e64_exp(a) + e64_exp(b) - 1023 + (int)n;
    return e64_double(((a ^ b) & 0x8000000000000000ull) | (((uint64_t)(e - 1) << 52) + hi + up));
}

// d^2 for the bits of d; ok is cleared where the square is not covered (a
// nonzero d whose square is not well inside the normal range).
LSM_HD double e64_sqr(uint64_t d, bool &ok)
{
    const bool zero = e64_zero(d);
    ok = ok && (zero || (unsigned)(e64_exp(d) - 520) < 1000u);
    return zero ? 0.0 : e64_prod(d, d);
}

// a b likewise (zero times a finite number is a signed zero).
LSM_HD double e64_mul(uint64_t a, uint64_t b, bool &ok)
{
    const bool zero = e64_zero(a) || e64_zero(b);
    ok = ok && (zero ? e64_exp(a) < 2047 && e64_exp(b) < 2047 : e64_prod_ok(a, b));
    return zero ? e64_double((a ^ b) & 0x8000000000000000ull) : e64_prod(a, b);
}

// a > b for doubles that are not negative (false for NaN), without the FP64
// pipe's comparison.
LSM_HD bool e64_gt(double a, double b)
{
    const uint64_t ua = e64_bits(a);
    return ua > e64_bits(b) && ua <= 0x7FF0000000000000ull;
}

#ifdef __CUDACC__
// The rare branches are calls: the compiler otherwise takes FP64 instructions,
// even a square root, out of such a branch and issues them every time.
static __device__ __noinline__ double e64_div_fp64(double a, double b) { return __ddiv_rn(a, b); }

struct Spring64 {
    double r2, e, f[3];
};

// A spring on the FP64 pipe (d[2] = 0 in 2D: adding +0 to the sum of two
// squares changes nothing).
static __device__ __noinline__ Spring64 e64_force_fp64(double dx, double dy, double dz, double k, double r0)
{
    Spring64 s;
    s.r2 = __dadd_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)), __dmul_rn(dz, dz));
    const double rd = __dsqrt_rn(s.r2);
    s.e = __dsub_rn(rd, r0);
    const double c = __ddiv_rn(__dmul_rn(k, s.e), rd);
    s.f[0] = __dmul_rn(c, dx);
    s.f[1] = __dmul_rn(c, dy);
    s.f[2] = __dmul_rn(c, dz);
    return s;
}

// x / m, correctly rounded; the usual unit mass costs nothing (x / 1 = x).
__device__ __forceinline__ double e64_div_mass(double x, double m)
{
    return e64_bits(m) == 0x3FF0000000000000ull ? x : e64_div_fp64(x, m);
}

// NS springs from their vectors d: r2 = |d|^2 (components in order), the
// stretch e = sqrt(r2) - r0, and the force f = ((k e) / sqrt(r2)) d on the lower
// end, every operation rounded as IEEE double. Left on the FP64 pipe: the sum of
// the squares and the subtraction of r0. Where an operand is outside the
// ranges above, all of that spring is done again there. The springs go through
// each stage together and without branches, so that their dependent chains
// (some 500 instructions each) overlap where few warps run.
template <int DIM, int NS>
__device__ __forceinline__ void e64_force_n(const double (&d)[NS][DIM], const double (&k)[NS], const double (&r0)[NS],
                                            double (&r2)[NS], double (&e)[NS], double (&f)[NS][DIM])
{
    bool ok[NS];
    Root64 r[NS];
#pragma unroll
    for (int s = 0; s < NS; s++) {
        ok[s] = true;
        r2[s] = e64_sqr(e64_bits(d[s][0]), ok[s]);
#pragma unroll
        for (int c = 1; c < DIM; c++) r2[s] = __dadd_rn(r2[s], e64_sqr(e64_bits(d[s][c]), ok[s]));
    }
#pragma unroll
    for (int s = 0; s < NS; s++) {
        const uint64_t x = e64_bits(r2[s]);
        ok[s] = ok[s] && (unsigned)((int)(x >> 52) - 1) < 2046u;  // positive and normal
        float y;
        asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(e64_sqrt_arg(x)));
        r[s] = e64_sqrt(x, y);
        e[s] = __dsub_rn(e64_root(r[s]), r0[s]);
    }
#pragma unroll
    for (int s = 0; s < NS; s++) {
        uint64_t ke = e64_bits(e[s]);
        if (NS > 1 || e64_bits(k[s]) != 0x3FF0000000000000ull) ke = e64_bits(e64_mul(e64_bits(k[s]), ke, ok[s]));
        const bool zero = e64_zero(ke);  // 0 / r = 0
        ok[s] = ok[s] && (zero || e64_div_ok(ke, r[s]));
        const uint64_t c = zero ? ke : e64_bits(e64_div(ke, r[s]));
#pragma unroll
        for (int q = 0; q < DIM; q++) f[s][q] = e64_mul(c, e64_bits(d[s][q]), ok[s]);
    }
#pragma unroll
    for (int s = 0; s < NS; s++)
        if (!ok[s]) {
            const Spring64 h = e64_force_fp64(d[s][0], d[s][1], DIM == 3 ? d[s][DIM - 1] : 0.0, k[s], r0[s]);
            r2[s] = h.r2;
            e[s] = h.e;
#pragma unroll
            for (int q = 0; q < DIM; q++) f[s][q] = h.f[q];
        }
}

// One spring.
template <int DIM>
__device__ __forceinline__ void e64_force(const double (&d)[DIM], double k, double r0, double &r2, double &e,
                                          double (&f)[DIM])
{
    double dn[1][DIM], fn[1][DIM], r2n[1], en[1];
    const double kn[1] = {k}, r0n[1] = {r0};
#pragma unroll
    for (int q = 0; q < DIM; q++) dn[0][q] = d[q];
    e64_force_n<DIM, 1>(dn, kn, r0n, r2n, en, fn);
    r2 = r2n[0];
    e = en[0];
#pragma unroll
    for (int q = 0; q < DIM; q++) f[q] = fn[0][q];
}
#endif

}  // namespace lsm
