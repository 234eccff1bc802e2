// df_pair.cuh -- two DF springs at a time on packed float instructions.
//
// The DF kernels are bound by instruction issue (strip kernel, 2048^2: 73% of
// the issue slots busy, FMA pipe 38%, ALU 45%), half of their instructions
// being FP32. sm_103a has add, mul and fma on pairs of floats (.f32x2): a packed
// instruction takes the FMA pipe as long as its two scalar ones, but one issue
// slot. spring_df_pair evaluates two springs side by side in the two halves;
// every element goes through the operations of spring_df (tile_body.cuh; 3D:
// spring3, tile3d.cu) in the same order with the same rounding, so both give the
// same bits. Differences and negations are written as fma with -1, exact like the
// subtraction.
// Together with the split force sums (DfSum) a 2048^2 step takes 89.1e6 warp
// instructions instead of 108.8e6 and 112.1 us instead of 122.8, a 256^3 foam's
// 830 us instead of 885 (775 on smaller blocks, tile3d.cu); what is left is
// spread over pipes (issue 65%, ALU 56%, FP64 53%, FMA 48%) at 20 warps per SM.
// F32 steps do the same (spring_f32_pair): 2048^2 90.5 -> 80.1 us, a 256^3
// foam 864 -> 714 (smaller blocks included).
#pragma once

#include "dfloat.cuh"

namespace lsm {

struct f32x2 {
    unsigned long long v;
};

__device__ __forceinline__ f32x2 pk(float a, float b)
{
    f32x2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(a), "f"(b));
    return r;
}

__device__ __forceinline__ void unpk(f32x2 p, float &a, float &b)
{
    asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(p.v));
}

__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b)
{
    f32x2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}

__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b)
{
    f32x2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}

__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c)
{
    f32x2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
    return r;
}

// A pair of double-floats.
struct ff2 {
    f32x2 hi, lo;
};

__device__ __forceinline__ f32x2 splat(float a) { return pk(a, a); }

// a - b
__device__ __forceinline__ f32x2 sub2(f32x2 a, f32x2 b) { return fma2(b, splat(-1.0f), a); }

__device__ __forceinline__ ff2 fast_two_sum2(f32x2 a, f32x2 b)
{
    const f32x2 s = add2(a, b);
    return ff2{s, sub2(b, sub2(s, a))};
}

__device__ __forceinline__ ff2 two_sum2(f32x2 a, f32x2 b)
{
    const f32x2 s = add2(a, b), bb = sub2(s, a);
    return ff2{s, add2(sub2(a, sub2(s, bb)), sub2(b, bb))};
}

// fix_to_ff_u24 of two values.
__device__ __forceinline__ ff2 fix_to_ff_u24_2(long long a, long long b)
{
    const int ha = (int)__funnelshift_r((unsigned)a, (unsigned)(a >> 32), 24);
    const int hb = (int)__funnelshift_r((unsigned)b, (unsigned)(b >> 32), 24);
    const f32x2 h = pk(__int2float_rn(ha), __int2float_rn(hb));
    const f32x2 l = mul2(pk(__int2float_rn((int)((unsigned)a & 0xFFFFFFu)), __int2float_rn((int)((unsigned)b & 0xFFFFFFu))),
                         splat(0x1p-24f));
    return fast_two_sum2(h, l);
}

// Two springs: vectors d[c][q], types t0, t1, whether they exist; M, cmax: the force
// split (TileArgs). Out: the split forces f[c][q] on the lower ends (zero where
// the spring does not exist or breaks now), the break test's outcome, and
// whether a force is beyond the split's exact range.
template <int DIM>
__device__ __forceinline__ void spring_df_pair(const long long (&d)[DIM][2], const TypeDF &t0, const TypeDF &t1,
                                               const bool (&live)[2], float M, float cmax, ff (&f)[DIM][2],
                                               bool (&brk)[2], bool &big)
{
    const f32x2 one = splat(1.0f), m1 = splat(-1.0f);
    ff2 x[DIM];
#pragma unroll
    for (int c = 0; c < DIM; c++) x[c] = fix_to_ff_u24_2(d[c][0], d[c][1]);
    // r^2 (ff_norm2_un, ff_norm3_un); names with n hold negated values
    f32x2 nx[DIM], p[DIM], ne[DIM];
#pragma unroll
    for (int c = 0; c < DIM; c++) {
        nx[c] = mul2(x[c].hi, m1);
        p[c] = mul2(x[c].hi, x[c].hi);
        ne[c] = fma2(nx[c], x[c].hi, p[c]);
    }
    ff2 s = two_sum2(p[0], p[1]);
    f32x2 nl = add2(ne[0], ne[1]);
    if constexpr (DIM == 3) {
        const ff2 t = two_sum2(s.hi, p[DIM - 1]);
        s = ff2{t.hi, add2(t.lo, s.lo)};
        nl = add2(nl, ne[DIM - 1]);
    }
#pragma unroll
    for (int c = 0; c < DIM; c++) nl = fma2(nx[c], add2(x[c].lo, x[c].lo), nl);
    const f32x2 nrl = sub2(nl, s.lo), nrh = mul2(s.hi, m1);  // -(r^2)
    float rh[2], nrlo[2];
    unpk(s.hi, rh[0], rh[1]);
    unpk(nrl, nrlo[0], nrlo[1]);
    brk[0] = live[0] && ff_gt_un(ff{rh[0], -nrlo[0]}, t0.rc2);
    brk[1] = live[1] && ff_gt_un(ff{rh[1], -nrlo[1]}, t1.rc2);
    // g = 1 - r0 / r (ff_spring_g)
    const f32x2 y = pk(rsqrt_approx(rh[0]), rsqrt_approx(rh[1])), ny = mul2(y, m1);
    const f32x2 q = mul2(y, y), nqe = fma2(ny, y, q);
    const f32x2 rho = fma2(nrl, q, fma2(s.hi, nqe, fma2(nrh, q, one)));
    const f32x2 r0h = pk(t0.r0.hi, t1.r0.hi), r0l = pk(t0.r0.lo, t1.r0.lo);
    const f32x2 py = mul2(r0h, y), npl = fma2(r0h, ny, py);
    const f32x2 t2 = fma2(mul2(py, splat(-0.5f)), fma2(mul2(rho, splat(0.75f)), rho, rho), fma2(r0l, ny, npl));
    const f32x2 g1 = fma2(py, m1, one);                // 1 - r0 y
    const f32x2 g2 = fma2(py, m1, fma2(g1, m1, one));  // its error: -r0 y - (g1 - 1)
    const ff2 g = fast_two_sum2(g1, add2(g2, t2));
    // c = k g (ff_mul_un)
    const f32x2 kh = pk(t0.k.hi, t1.k.hi);
    const f32x2 cc = mul2(kh, g.hi);
    const f32x2 cr = fma2(pk(t0.k.lo, t1.k.lo), g.hi, fma2(kh, g.lo, fma2(kh, g.hi, mul2(cc, m1))));
    float c0, c1, l0, l1;
    unpk(cc, c0, c1);
    unpk(cr, l0, l1);
    const bool on0 = live[0] && !brk[0], on1 = live[1] && !brk[1];
    c0 = on0 ? c0 : 0.0f;
    c1 = on1 ? c1 : 0.0f;
    big |= fmaxf(fabsf(c0), fabsf(c1)) > cmax;
    const f32x2 ch = pk(c0, c1), nch = mul2(ch, m1), cl = pk(on0 ? l0 : 0.0f, on1 ? l1 : 0.0f);
    // the split products (ff_mul_split)
    const f32x2 M2 = splat(M), nM2 = splat(-M);
#pragma unroll
    for (int c = 0; c < DIM; c++) {
        const f32x2 fq = add2(fma2(nch, x[c].hi, M2), nM2);
        const f32x2 fe = fma2(cl, x[c].hi, fma2(ch, x[c].lo, fma2(ch, x[c].hi, fq)));
        unpk(fq, f[c][0].hi, f[c][1].hi);
        unpk(fe, f[c][0].lo, f[c][1].lo);
    }
}

// Two F32 springs: e[c][q], the vectors minus their lattice vectors (o[c][q], oo =
// |o|^2) in fixed point; types t = (k, r0, rc2, cor); whether they exist. Out: the
// forces on the lower ends and the break test's outcome. The operations of
// spring_f32_o (tile_body.cuh) and spring3 (tile3d.cu); the terms of r^2 - r0^2 are
// added to cor in their order: y, x in 2D, x, y, z in 3D.
template <int DIM>
__device__ __forceinline__ void spring_f32_pair(const long long (&e)[DIM][2], const f32x2 (&o)[DIM], f32x2 oo,
                                                const float4 &t0, const float4 &t1, const bool (&live)[2], float p24,
                                                float p0, float (&f)[DIM][2], bool (&brk)[2])
{
    f32x2 x[DIM];
#pragma unroll
    for (int c = 0; c < DIM; c++) {
        const f32x2 h = pk(__int2float_rn((int)(e[c][0] >> 24)), __int2float_rn((int)(e[c][1] >> 24)));
        const f32x2 l = pk(__int2float_rn((int)(e[c][0] & 0xFFFFFFLL)), __int2float_rn((int)(e[c][1] & 0xFFFFFFLL)));
        x[c] = fma2(h, splat(p24), mul2(l, splat(p0)));
    }
    const f32x2 two = splat(2.0f);
    f32x2 num = pk(t0.w, t1.w);
#pragma unroll
    for (int q = 0; q < DIM; q++) {
        const int c = DIM == 2 ? 1 - q : q;
        num = fma2(fma2(o[c], two, x[c]), x[c], num);  // (2 o + e) e: the doubling is exact
    }
    const f32x2 r2 = add2(oo, num);
    float a, b, na, nb;
    unpk(r2, a, b);
    unpk(num, na, nb);
    brk[0] = live[0] && a > t0.z;
    brk[1] = live[1] && b > t1.z;
    const f32x2 ir = pk(rsqrt_approx(a), rsqrt_approx(b));
    float da, db;
    unpk(fma2(r2, ir, pk(t0.y, t1.y)), da, db);
    const f32x2 s = pk(__fdividef(na, da), __fdividef(nb, db));  // r - r0
    float ca, cb;
    unpk(mul2(mul2(pk(t0.x, t1.x), s), ir), ca, cb);
    const f32x2 k = pk(live[0] && !brk[0] ? ca : 0.0f, live[1] && !brk[1] ? cb : 0.0f);
#pragma unroll
    for (int c = 0; c < DIM; c++) unpk(mul2(k, add2(o[c], x[c])), f[c][0], f[c][1]);
}

}  // namespace lsm
