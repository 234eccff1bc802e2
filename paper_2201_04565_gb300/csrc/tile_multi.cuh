// tile_multi.cuh -- several time steps of a TX x TY tile in one launch, for 2D
// images too small to fill the device.
//
// What bounds such a step is not work but a chain: the launch, the loads of the
// state, four springs and a gather one after another in each thread, the
// stores. A block therefore takes its tile with a halo of H cells, keeps the
// state of every cell of that region in the registers of G threads, and runs
// up to H time steps on it before it writes its own cells back. The cells of
// the halo are computed like its own and lose one ring per step, so no block
// waits for another within the launch.
//   - One cell per thread (or G threads per cell, which share its four forward
//     springs and its two components): no loop over rows, and a thread's
//     springs go side by side (spring_df, spring_f32, e64_force_n), so their
//     dependent chains overlap.
//   - Per step: drift, positions to shared memory; barrier; springs, forces to
//     shared memory; barrier; the gather in the canonical order and the
//     half-kicks. Every floating-point operation is the one-step tile kernel's,
//     in the same order: positions, velocities, broken flags and break steps
//     are the same bits.
//   - SAMPLE: the last step of the launch also writes v(t + dt) and the tile's
//     partial sums of the sample (grouped per tile of this kernel).
//   - Broken flags: a halo cell's flag may be set by its owner during this very
//     launch, at a later one of its steps, before this block reads it. Its break
//     step tells (it is written by the owner too, and is not below this
//     launch's first step, or not yet there): such a break is left to this
//     block's own break test, which comes to the same decision at its step.
// The chain costs about 1.2 us per launch and 1.7 us per step (100 x 90, DF), so
// a halo of 3 on 16 x 4 tiles takes the step from 5.5 to 2.2 us there; what the
// halo repeats (2.1 times the tile's work for that shape, 1.3 times for 32 x 8
// cells and a halo of 2) is what larger images cannot afford. See multi_shape
// (tile_multi.cu) for where the lines lie.
#pragma once

#include "df_pair.cuh"
#include "tile_body.cuh"

namespace lsm {

// Region of a tile: its TX x TY cells and a halo of H; G threads per cell.
template <int TX, int TY, int H, int G>
struct MultiShape {
    static constexpr int RX = TX + 2 * H, RY = TY + 2 * H, N = RX * RY;
    static constexpr int NP = (N + 31) / 32 * 32, NT = G * NP, NW = NT / 32;
};

template <int PREC>
using multi_force = typename std::conditional<PREC == LSM_PREC_F32, float,
                    typename std::conditional<PREC == LSM_PREC_DF, ff, double>::type>::type;

template <int TX, int TY, int H, int G, int PREC>
constexpr size_t multi_smem_bytes()
{
    return (size_t)MultiShape<TX, TY, H, G>::N * (16 + 8 * sizeof(multi_force<PREC>) + 1) + 16;
}

// ns (1..H) time steps of tile (bx, by); tile_id indexes the partial sums.
template <int TX, int TY, int H, int G, int PREC, bool RATE, bool SAMPLE>
__device__ __forceinline__ void tile_multi_body(const TileArgs &A, int bx, int by, int64_t tile_id, int ns,
                                                unsigned char *smem_raw)
{
    using M = MultiShape<TX, TY, H, G>;
    constexpr bool FIX = PREC == LSM_PREC_F32 || PREC == LSM_PREC_DF;
    using FT = multi_force<PREC>;
    using PT = typename std::conditional<FIX, long long, double>::type;
    using AT = typename std::conditional<FIX, ff, double>::type;  // sample sums
    constexpr int RX = M::RX, RY = M::RY, N = M::N, NP = M::NP, NT = M::NT, NW = M::NW;
    constexpr int NS = 4 / G;              // springs per thread
    constexpr int NC = G == 1 ? 2 : 1;     // components per thread (groups 0 and 1 when G > 1)
    PT *sx = (PT *)smem_raw;               // [2][N] drifted positions
    FT *sf = (FT *)(sx + 2 * N);           // [2][4][N] forces on the lower ends
    uint8_t *sph = (uint8_t *)(sf + 8 * N);
    __shared__ SpringType stab[FIX ? 1 : 128];
    __shared__ TypeDF sdf[FIX ? 128 : 1];
    __shared__ ff soff[4][3];
    __shared__ double sred[SAMPLE ? 6 : 1][NW];

    const int tid = threadIdx.x;
    const int grp = G == 1 ? 0 : tid / NP;  // warp-uniform
    const int e = tid - grp * NP;
    const int rx = e % RX, ry = e / RX;
    const int gx = bx * TX - H + rx, gy = by * TY - H + ry;
    const bool in = e < N && gx >= 0 && gx < A.nx && gy >= 0 && gy < A.ny;
    // the cell is right up to this step of the launch (its distance to the edge)
    const int depth = e < N ? min(min(rx, RX - 1 - rx), min(ry, RY - 1 - ry)) : -1;
    const int64_t g = (int64_t)gy * A.nx + gx;
    const bool comps = G == 1 || grp < 2;  // this thread moves components c0 .. c0 + NC - 1
    const int c0 = G == 1 ? 0 : grp;
    unsigned ph = 0, mk = 0;
    double p[NC], v[NC];
#pragma unroll
    for (int c = 0; c < NC; c++) p[c] = v[c] = 0.0;
    if (in) {
        ph = A.phase[g];
        mk = A.mask[g];
        if (comps) {
#pragma unroll
            for (int c = 0; c < NC; c++) {
                p[c] = A.x_in[(c0 + c) * A.np + g];
                v[c] = A.vh_in[(c0 + c) * A.np + g];
            }
        }
    }
    const int nt = 2 * A.nphase * A.nphase;
    for (int q = tid; q < nt; q += NT) {
        if constexpr (FIX) sdf[q] = A.tdf[q];
        else stab[q] = A.types[q];
    }
    if (PREC == LSM_PREC_F32 && tid < 4) {
        const int dx = tid == 0 ? 1 : (tid == 1 ? -1 : (tid == 2 ? 0 : 1));
        const int dy = tid == 0 ? 0 : 1;
        const ff ox = fix_to_ff((long long)dx * A.a_fix, A.S), oy = fix_to_ff((long long)dy * A.a_fix, A.S);
        soff[tid][0] = ox;
        soff[tid][1] = oy;
        soff[tid][2] = ff_add(ff_mul(ox, ox), ff_mul(oy, oy));
    }
    if (grp == 0 && e < N) sph[e] = (uint8_t)ph;
    const bool grip = gx == 0 || gx == A.nx - 1;
    const bool own = in && rx >= H && rx < H + TX && ry >= H && ry < H + TY && ph;
    const long long step0 = *A.d_step + A.t_off;
    double m = 1.0;
    Coef4 k4{};
    if (ph) {
        if (PREC == LSM_PREC_EXACT64 || SAMPLE) m = A.mass[ph - 1];
        if constexpr (FIX) k4 = A.coef[ph - 1];
    }
    // a neighbour's cells: only breaks of earlier launches count (see above)
    if (!own && mk) {
        unsigned old = 0;
#pragma unroll
        for (int q = 0; q < NS; q++) {
            const int slot = grp * NS + q;
            if ((mk >> slot) & 1) {
                const long long b = A.brk[(int64_t)slot * A.np + g];
                if (b >= 0 && b < step0) old |= 1u << slot;
            }
        }
        mk = old;
    }
    bool over = false, bad = false;
    AT w_acc{}, u_acc{}, react{};
    double mvx2 = 0.0, ke = 0.0, res = 0.0;
    float mvx2f = 0.0f, kef = 0.0f, resf = 0.0f;
    __syncthreads();

#pragma unroll 1
    for (int s = 0; s < ns; s++) {
        const bool last = SAMPLE && s == ns - 1;
        // drift
        if (comps && ph && depth >= s) {
#pragma unroll
            for (int c = 0; c < NC; c++) {
                const bool fixed = grip && (c0 + c == 0 || A.grip_mode == 1);
                if (RATE && grip && c0 + c == 0) {
                    const long long st = step0 + s + 1 - A.rate_step0;
                    const double X = ml((double)gx, A.a);
                    p[c] = ad(X, ml(ad(A.rate_eps0, ml((double)st, A.rate_dt)), sb(X, A.xc)));
                }
                if constexpr (FIX) {
                    if (!fixed) p[c] = fma(A.dt, v[c], p[c]);
                    sx[(c0 + c) * N + e] = dbl_to_fix(p[c], A.S, over);
                } else {
                    if (!fixed) p[c] = ad(p[c], ml(A.dt, v[c]));
                    sx[(c0 + c) * N + e] = p[c];
                }
            }
        }
        __syncthreads();
        // forward springs: a thread's are evaluated without branches between
        // them (one that is not there is computed on whatever its cells hold
        // and dropped), so that their dependent chains overlap
        FT fx[NS], fy[NS];
        unsigned nb = 0;
        bool big = false;  // DF: a force beyond the split's exact range
        if (ph && depth >= s) {
            unsigned live = 0, longer = 0;
            int ti[NS], qq[NS];
#pragma unroll
            for (int q = 0; q < NS; q++) {
                const int slot = grp * NS + q;
                const int dq = slot == 0 ? 1 : RX - 2 + slot;
                qq[q] = min(e + dq, N - 1);
                const unsigned pq = sph[qq[q]];
                if (pq && !((mk >> slot) & 1)) live |= 1u << q;
                ti[q] = pq ? (((int)(ph - 1) * A.nphase) + (int)(pq - 1)) * 2 + (slot & 1) : 0;
            }
            const PT mx = sx[e], my = sx[N + e];
            if constexpr (PREC == LSM_PREC_EXACT64) {
                double dd[NS][2], k[NS], r0[NS], r2[NS], st[NS], f[NS][2];
#pragma unroll
                for (int q = 0; q < NS; q++) {
                    dd[q][0] = sb(sx[qq[q]], mx);
                    dd[q][1] = sb(sx[N + qq[q]], my);
                    k[q] = stab[ti[q]].k;
                    r0[q] = stab[ti[q]].r0;
                }
                e64_force_n<2, NS>(dd, k, r0, r2, st, f);
#pragma unroll
                for (int q = 0; q < NS; q++) {
                    if (e64_gt(r2[q], stab[ti[q]].rc2)) longer |= 1u << q;
                    fx[q] = f[q][0];
                    fy[q] = f[q][1];
                    if (last && own && ((live & ~longer) >> q) & 1) {
                        u_acc += ml(ml(ml(0.5, k[q]), st[q]), st[q]);
                        w_acc += ml(dd[q][0], f[q][0]);
                    }
                }
            } else if constexpr (PREC == LSM_PREC_DF && !SAMPLE) {  // two springs at a time
#pragma unroll
                for (int q = 0; q < NS; q += 2) {
                    const long long dd[2][2] = {{sx[qq[q]] - mx, sx[qq[q + 1]] - mx},
                                                {sx[N + qq[q]] - my, sx[N + qq[q + 1]] - my}};
                    const bool lv[2] = {(bool)((live >> q) & 1), (bool)((live >> (q + 1)) & 1)};
                    ff f[2][2];
                    bool brk[2];
                    spring_df_pair<2>(dd, sdf[ti[q]], sdf[ti[q + 1]], lv, A.df_M, A.df_cmax, f, brk, big);
#pragma unroll
                    for (int h = 0; h < 2; h++) {
                        if (brk[h]) longer |= 1u << (q + h);
                        fx[q + h] = f[0][h];
                        fy[q + h] = f[1][h];
                    }
                }
            } else {
#pragma unroll
                for (int q = 0; q < NS; q++) {
                    const PT dx = sx[qq[q]] - mx, dy = sx[N + qq[q]] - my;
                    const TypeDF t = sdf[ti[q]];
                    FT dxf, st;
                    if constexpr (PREC == LSM_PREC_F32) {
                        if (spring_f32<true, SAMPLE>(dx, dy, grp * NS + q, t, soff, A, fx[q], fy[q], dxf, st))
                            longer |= 1u << q;
                    } else {
                        if (ff_gt_un(ff_norm2_un(fix_to_ff_u24(dx), fix_to_ff_u24(dy)), t.rc2)) longer |= 1u << q;
                        spring_df<false, SAMPLE>(dx, dy, t, A, fx[q], fy[q], dxf, st, big);
                    }
                    if (last && own && ((live & ~longer) >> q) & 1) {
                        if constexpr (PREC == LSM_PREC_F32) {
                            u_acc = ff_add_f(u_acc, 0.5f * t.k.hi * st * st);
                            w_acc = ff_add_f(w_acc, dxf * fx[q]);
                        } else if constexpr (PREC == LSM_PREC_DF) {
                            u_acc = ff_add_sloppy(u_acc, ff_mul(ff_mul_f(t.k, 0.5f), ff_sqr(st)));
                            w_acc = ff_add_sloppy(w_acc, ff_mul(dxf, df_pair(fx[q])));
                        }
                    }
                }
            }
            nb = live & longer;
#pragma unroll
            for (int q = 0; q < NS; q++)
                if (!(((live & ~longer) >> q) & 1)) fx[q] = fy[q] = FT{};
        } else {
#pragma unroll
            for (int q = 0; q < NS; q++) fx[q] = fy[q] = FT{};
        }
        if (e < N) {
#pragma unroll
            for (int q = 0; q < NS; q++) {
                sf[(grp * NS + q) * N + e] = fx[q];
                sf[(4 + grp * NS + q) * N + e] = fy[q];
            }
        }
        if (nb) {
            nb <<= grp * NS;
            mk |= nb;
            if (own) {
                // the groups of a cell share its flag byte (tile_mask_bytes: whole words)
                const uintptr_t a = (uintptr_t)(A.mask + g);
                atomicOr((unsigned *)(a & ~(uintptr_t)3), nb << (8 * (a & 3)));
#pragma unroll
                for (int slot = 0; slot < 4; slot++)
                    if ((nb >> slot) & 1) {
                        A.brk[(int64_t)slot * A.np + g] = step0 + s;
                        atomicMin(A.first_break, (unsigned long long)(step0 + s));
                        atomicAdd(A.nbroken, 1ull);
                    }
            }
        }
        bool careful = false;
        if constexpr (PREC == LSM_PREC_DF) careful = __syncthreads_or(big);
        else __syncthreads();
        // gather and integrate
        if (comps && ph && depth > s) {
#pragma unroll
            for (int c = 0; c < NC; c++) {
                const FT *f = sf + (c0 + c) * 4 * N + e;
                const FT i3 = f[3 * N - RX - 1], i2 = f[2 * N - RX], i1 = f[N - RX + 1], i0 = f[-1];
                double F;
                float Ff = 0.0f;
                ff Fd{0.0f, 0.0f};
                if constexpr (PREC == LSM_PREC_EXACT64) {
                    F = sb(sb(sb(sb(0.0, i3), i2), i1), i0);
                    F = ad(ad(ad(ad(F, f[0]), f[N]), f[2 * N]), f[3 * N]);
                } else if constexpr (PREC == LSM_PREC_DF) {
                    DfSum acc;
                    if (!careful) acc = df_gather<DfSum>(i3, i2, i1, i0, f, N);
                    else acc = df_gather<DfSumCareful>(i3, i2, i1, i0, f, N);
                    F = acc.value(A.df_bias);
                    Ff = __fmul_rn(__fadd_rn(acc.hs, acc.el), A.p24);  // back from units of 2^(24-S)
                    Fd = ff{acc.hs, acc.el};                            // (in those units)
                } else {
                    float acc = f[0] - i3;
                    acc += f[N] - i2;
                    acc += f[2 * N] - i1;
                    acc += f[3 * N] - i0;
                    F = f2d_force(acc);
                    Ff = acc;
                    Fd = ff{acc, 0.0f};
                }
                if (last && own && c0 + c == 0 && gx == A.nx - 1) {  // right-grip reaction
                    if constexpr (FIX) react = ff_neg(Fd);
                    else react = sb(0.0, F);
                }
                if (grip && (c0 + c == 0 || A.grip_mode == 1)) {
                    v[c] = 0.0;
                    if (last && own) A.v_obs[(c0 + c) * A.np + g] = 0.0;
                    continue;
                }
                double vn = 0.0;
                if constexpr (PREC == LSM_PREC_EXACT64) {
                    const double acc = e64_div_mass(sb(F, ml(A.gamma, v[c])), m);
                    vn = ad(v[c], ml(A.hdt, acc));
                    v[c] = ad(vn, ml(A.hdt, acc));
                } else {
                    if (last) vn = fma(k4.c2h, F, k4.c1h * v[c]);
                    v[c] = fma(k4.c2, F, k4.c1 * v[c]);
                }
                if (last && own) {
                    A.v_obs[(c0 + c) * A.np + g] = vn;
                    bad |= !dbl_finite_bits(vn) || !dbl_finite_bits(p[c]);
                    if constexpr (FIX) {
                        const float vf = d2f_bits(vn), mf = (float)m;
                        resf = fmaxf(resf, fmaxf(fabsf(Ff), fabsf(vf)));
                        kef = fmaf(0.5f * mf * vf, vf, kef);
                        if (c0 + c == 0) mvx2f = mf * vf * vf;
                    } else {
                        res = fmax(res, fmax(fabs(F), fabs(vn)));
                        ke += 0.5 * m * vn * vn;
                        if (c0 + c == 0) mvx2 = m * vn * vn;
                    }
                }
            }
        }
    }
    if (FIX && over) atomicOr(A.status, 2);
    if (own && comps) {
#pragma unroll
        for (int c = 0; c < NC; c++) {
            A.x_out[(c0 + c) * A.np + g] = p[c];
            A.vh_out[(c0 + c) * A.np + g] = v[c];
        }
    }
    if constexpr (SAMPLE) {
        if (bad) atomicOr(A.status, 1);
        // the six sums of the sample: warp trees side by side, then one
        // thread per sum over the warps
        double t[6];
        if constexpr (FIX) {
            ff q[5] = {w_acc, u_acc, ff{mvx2f, 0.0f}, ff{kef, 0.0f}, react};
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
#pragma unroll
                for (int k = 0; k < 5; k++)
                    q[k] = ff_add_sloppy(q[k], ff{__shfl_xor_sync(0xffffffffu, q[k].hi, o),
                                                  __shfl_xor_sync(0xffffffffu, q[k].lo, o)});
                resf = fmaxf(resf, __shfl_xor_sync(0xffffffffu, resf, o));
            }
            if ((tid & 31) == 0) {
#pragma unroll
                for (int k = 0; k < 5; k++) t[k] = ff_to_double(q[k]);
                t[5] = f2d_bits(resf);
            }
        } else {
            t[0] = w_acc;
            t[1] = u_acc;
            t[2] = mvx2;
            t[3] = ke;
            t[4] = react;
            t[5] = res;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
#pragma unroll
                for (int k = 0; k < 5; k++) t[k] += __shfl_xor_sync(0xffffffffu, t[k], o);
                t[5] = fmax(t[5], __shfl_xor_sync(0xffffffffu, t[5], o));
            }
        }
        if ((tid & 31) == 0)
#pragma unroll
            for (int k = 0; k < 6; k++) sred[k][tid >> 5] = t[k];
        __syncthreads();
        if (tid < 6) {
            double r = 0.0;
            for (int w = 0; w < NW; w++) r = tid == 5 ? fmax(r, sred[5][w]) : r + sred[tid][w];
            if (PREC == LSM_PREC_DF) {  // from units of 2^(24-S) (exact)
                const double u = (double)A.p24;
                if (tid < 2) r *= u * u;
                if (tid == 4) r *= u;
            }
            if (tid < 2) A.part_s[tid * A.ntiles + tile_id] = r;
            else A.part_p[(tid - 2) * A.ntiles + tile_id] = r;
        }
    }
}

}  // namespace lsm
