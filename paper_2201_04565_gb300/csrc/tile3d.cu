// tile3d.cu -- one launch per time step for 3D voxel lattices (first and
// second neighbours, 18 springs per interior particle) in the fixed-point
// modes (F32, DF).
//
// A CTA (256 threads) owns a 16 x 8 x 8 block of voxels. Per time step it
//   1. loads the block plus a one-voxel halo (phase, broken flags, positions
//      drifted by dt vh, Eq. 3) into shared memory as 64-bit fixed point, and
//      writes the block's own drifted positions, x(t+dt);
//   2. compacts the block's particles into a list in raster order (porous
//      volumes leave most voxels void; the list keeps every warp busy);
//   3. for each listed particle evaluates all 18 of its springs slot by slot
//      (forward offsets by ascending target), the incoming spring then the
//      outgoing one, accumulating the force in registers: not the canonical
//      order of the sequential sum, but the same in every step, so that the
//      states do not depend on how the steps are grouped into calls. Every
//      spring is evaluated by both endpoints from the same data (d = x_upper
//      - x_lower, the upper endpoint negates the force), so both see the same
//      break decision and equal and opposite forces; the lower endpoint
//      records breaks. No shared-memory force exchange: in 3D that (9 slots x
//      3 components per source voxel) would cost more shared memory than the
//      recomputation costs arithmetic in these modes;
//      and integrates (Eqs. 4-5) in FP64, writing vh(t+3dt/2).
// The FP64 modes keep the spring-list kernels for 3D: recomputing every
// spring twice would double their FP64-pipe work.
//
// Broken flags: 9 bits per voxel (its forward springs in slot order, the
// canonical order of the targets), written only by the owning thread; break
// steps [9][nv].
#include "df_pair.cuh"
#include "tile_body.cuh"

#include <algorithm>
#include <cmath>
#include <vector>

namespace lsm {

namespace {

// 16 x 8 x 8 blocks, four CTAs of 256 threads per SM (51 KB and 64 registers each):
// one CTA's region load runs beside the others' springs. Against 32 x 8 x 8 blocks
// in two CTAs of 512 the halo is a little dearer (1.76 region voxels per voxel,
// 1.66) and the 256^3 foam's step 830 -> 775 us; 32 x 8 x 4 in three of 256: 816;
// 16 x 8 x 4 in six of 128: 794. Writing the drifted positions as they are loaded
// (the integration no longer reads x and vh's drift again) and one warp scanning
// the row counts take it to 754. Without the springs it takes 400: region loads
// cost as much as arithmetic. Listing the region's particles first and loading
// only those, two at a time, has the same instructions and more barriers (831);
// two voxels' state in flight per thread spills (768).
constexpr int T3X = 16, T3Y = 8, T3Z = 8, T3V = T3X * T3Y * T3Z;  // voxels per block
constexpr int T3N = 256;                                           // threads per CTA
constexpr int T3MIN = 4;                                           // CTAs per SM
constexpr int R3X = T3X + 2, R3Y = T3Y + 2, R3Z = T3Z + 2, R3N = R3X * R3Y * R3Z;

// shared memory of one CTA (dynamic)
struct Smem3 {
    long long xf[3][R3N];     // fixed-point drifted positions of the region
    uint16_t mk[R3N];         // broken flags
    uint16_t list[T3V];       // region indices of the block's particles (compacted)
    uint8_t ph[R3N];          // phase (0 = void)
};

struct Tile3Args {
    int nx, ny, nz, nphase;
    int64_t nv;
    const double *x_in, *vh_in;
    double *x_out, *vh_out, *v_obs;
    const uint8_t *phase;
    uint16_t *mask;
    long long *brk;  // [9][nv]
    const TypeDF *tdf;
    const double *mass;
    const Coef4 *coef;
    int S;
    long long a_fix;
    float p24, p0;
    double dt, a, xc;
    int grip_mode;
    int rate_on;  // constant strain rate: grips at rate_eps0 + (s - rate_step0) rate_dt
    double rate_eps0, rate_dt;
    long long rate_step0;
    const long long *d_step;
    int64_t t_off;
    unsigned long long *first_break, *nbroken;
    int *status;
    double *part_s, *part_p;
    int64_t ntiles;
    int sd[9][3];   // forward offsets in canonical (ascending raster) order
    int ssh[9];     // their shells (1: face, 2: edge diagonal)
    float oo2[2];   // |o|^2 per shell as floats (F32 mode)
    float fa;       // lattice spacing as a float (F32 mode)
    unsigned df_bias;     // DF: as TileArgs
    float df_M, df_cmax;
};

// x of a grip at the strain of the step being computed (constant strain
// rate); the kernel evaluates it for the two grip columns once per thread
__device__ __forceinline__ double rate_grip_x(const Tile3Args &A, int gx)
{
    const long long s = *A.d_step + A.t_off + 1 - A.rate_step0;
    const double eps = __dadd_rn(A.rate_eps0, __dmul_rn((double)s, A.rate_dt));
    const double X = __dmul_rn((double)gx, A.a);
    return __dadd_rn(X, __dmul_rn(eps, __dsub_rn(X, A.xc)));
}

// Whether region voxel e belongs to the block itself (not to its halo).
__device__ __forceinline__ bool in_block(int e)
{
    const int rx = e % R3X, ry = (e / R3X) % R3Y, rz = e / (R3X * R3Y);
    return rx >= 1 && rx <= T3X && ry >= 1 && ry <= T3Y && rz >= 1 && rz <= T3Z;
}

// A region voxel on its way from memory to shared memory (g < 0: outside).
struct RawVoxel {
    int64_t g;
    uint8_t ph;
};

__device__ __forceinline__ RawVoxel voxel_at(const Tile3Args &A, int x0, int y0, int z0, int e)
{
    const int gx = x0 - 1 + e % R3X, gy = y0 - 1 + (e / R3X) % R3Y, gz = z0 - 1 + e / (R3X * R3Y);
    RawVoxel r{-1, 0};
    if (gx >= 0 && gx < A.nx && gy >= 0 && gy < A.ny && gz >= 0 && gz < A.nz) {
        r.g = gx + (int64_t)A.nx * (gy + (int64_t)A.ny * gz);
        r.ph = A.phase[r.g];
    }
    return r;
}

// rate_l, rate_r: the grips' x under the constant strain rate (RATE); own: a
// voxel of the block itself, whose drifted position is the step's output
template <int MODE, bool SAMPLE, bool RATE>
__device__ __forceinline__ void load_voxel(const Tile3Args &A, int x0, int e, const RawVoxel &r, Smem3 &S, bool &over,
                                           bool &bad, double rate_l, double rate_r)
{
    uint16_t mk = 0;
    double px[3] = {0.0, 0.0, 0.0};
    if (r.ph) {
        const int gx = x0 - 1 + e % R3X;
        mk = A.mask[r.g];
        const bool grip = gx == 0 || gx == A.nx - 1;
#pragma unroll
        for (int c = 0; c < 3; c++) {
            px[c] = A.x_in[c * A.nv + r.g];
            const bool fixed = grip && (c == 0 || A.grip_mode == 1);
            if (MODE == T_STEP && !fixed) px[c] = fma(A.dt, A.vh_in[c * A.nv + r.g], px[c]);
        }
        if (RATE && MODE == T_STEP && grip) px[0] = gx == 0 ? rate_l : rate_r;
        if (MODE == T_STEP && in_block(e)) {
#pragma unroll
            for (int c = 0; c < 3; c++) {
                A.x_out[c * A.nv + r.g] = px[c];
                if (SAMPLE && !(grip && (c == 0 || A.grip_mode == 1))) bad |= !dbl_finite_bits(px[c]);
            }
        }
#pragma unroll
        for (int c = 0; c < 3; c++) S.xf[c][e] = dbl_to_fix(px[c], A.S, over);
    }
    S.ph[e] = r.ph;
    S.mk[e] = mk;
}

// Force of the spring lower -> upper on the lower endpoint (d = x_upper -
// x_lower); false if the spring breaks now (r^2 > rc^2).
template <int PREC, bool TEST>
__device__ __forceinline__ bool spring3(const Tile3Args &A, const long long *dl, const long long *du, int s,
                                        const TypeDF &t, ff *f, ff &w, ff &u, bool sample)
{
    if constexpr (PREC == LSM_PREC_DF) {  // lengths in units of 2^(24-S), as spring_df
        ff d[3];
#pragma unroll
        for (int c = 0; c < 3; c++) d[c] = fix_to_ff_u24(du[c] - dl[c]);
        const ff r2 = ff_norm3_un(d[0], d[1], d[2]);
        if (TEST && ff_gt_un(r2, t.rc2)) return false;
        ff y;
        const ff g = ff_spring_g(r2, t.r0, sample ? &y : nullptr);
        const ff cc = ff_mul_un(t.k, g);  // unnormalised: only multiplied further
#pragma unroll
        for (int c = 0; c < 3; c++) f[c] = ff_mul_split(cc, d[c], A.df_M);
        if (sample) {  // double-float sums: no FP64 pipe work per spring
            const ff st = ff_mul(ff_mul(r2, y), g);  // r - r0
            u = ff_add_sloppy(u, ff_mul(ff_mul_f(t.k, 0.5f), ff_sqr(st)));
            w = ff_add_sloppy(w, ff_mul(d[0], df_pair(f[0])));
        }
    } else {  // F32: e = d - o exact, (2 o + e).e carries no cancellation; the operations of spring_f32_pair
        float e[3], dd[3], num = t.cor.hi;
#pragma unroll
        for (int c = 0; c < 3; c++) {
            const long long ef = du[c] - dl[c] - (long long)A.sd[s][c] * A.a_fix;
            e[c] = fix_to_float_i2f(ef, A.p24, A.p0);
            const float o = A.sd[s][c] == 0 ? 0.0f : (A.sd[s][c] > 0 ? A.fa : -A.fa);
            dd[c] = __fadd_rn(o, e[c]);
            num = __fmaf_rn(__fmaf_rn(o, 2.0f, e[c]), e[c], num);
        }
        const float r2f = __fadd_rn(A.oo2[A.ssh[s] - 1], num);
        if (TEST && r2f > t.rc2.hi) return false;
        const float ir = rsqrt_approx(r2f);
        const float st = __fdividef(num, __fmaf_rn(r2f, ir, t.r0.hi));  // r - r0
        const float cc = __fmul_rn(__fmul_rn(t.k.hi, st), ir);
#pragma unroll
        for (int c = 0; c < 3; c++) f[c] = ff{-__fmul_rn(cc, dd[c]), 0.0f};  // in the form of a split force
        if (sample) {
            u = ff_add_f(u, 0.5f * t.k.hi * st * st);
            w = ff_add_f(w, dd[0] * -f[0].hi);
        }
    }
    return true;
}

// The 18 springs of a particle: forces into F (split sums), new breaks of its
// forward springs into newb; slot s's incoming spring is broken by its source's
// flags or its own break test, which the source's thread records. Slot by slot, the
// incoming spring then the outgoing one: they share offset, shell and lattice vector.
// (Pairs in the canonical order, all incoming springs first, took the 256^3 foam
// from 755 to 781 us a step, in F32 from 697 to 770.) In DF the sums
// go without error terms until a factor above cmax turns up (up to then every
// partial sum is exact, see DfSum), and with them from there on. (Running all 18
// springs again with error terms instead took the 256^3 foam from 754 to 970 us
// a step at 10% compression, 797 this way.)
template <int PREC>
__device__ __forceinline__ void tile3_pairs(const Tile3Args &A, const Smem3 &S, const TypeDF *sdf, const int *soff,
                                            int ep, int pp, uint16_t mk, const long long (&xp)[3], DfSumCareful (&F)[3],
                                            uint16_t &newb)
{
    bool big = PREC != LSM_PREC_DF;  // F32's forces are plain floats: always with error terms
#pragma unroll 1
    for (int s = 0; s < 9; s++) {
        const int o = soff[s], ei = ep - o, eo = ep + o, sh = A.ssh[s] - 1;
        const int pi = S.ph[ei], po = S.ph[eo];
        const bool live[2] = {pi && !((S.mk[ei] >> s) & 1), po && !((mk >> s) & 1)};
        if (!live[0] && !live[1]) continue;
        const TypeDF &ti = sdf[live[0] ? (((pi - 1) * A.nphase) + (pp - 1)) * 2 + sh : 0];
        const TypeDF &to = sdf[live[1] ? (((pp - 1) * A.nphase) + (po - 1)) * 2 + sh : 0];
        long long d[3][2];
#pragma unroll
        for (int c = 0; c < 3; c++) {
            d[c][0] = xp[c] - S.xf[c][ei];
            d[c][1] = S.xf[c][eo] - xp[c];
        }
        ff f[3][2];
        bool brk[2];
        if constexpr (PREC == LSM_PREC_DF) {
            spring_df_pair<3>(d, ti, to, live, A.df_M, A.df_cmax, f, brk, big);
        } else {
            f32x2 o3[3];
#pragma unroll
            for (int c = 0; c < 3; c++) {
                const int k = A.sd[s][c];
                d[c][0] -= (long long)k * A.a_fix;
                d[c][1] -= (long long)k * A.a_fix;
                o3[c] = splat(k == 0 ? 0.0f : (k > 0 ? A.fa : -A.fa));
            }
            float ff3[3][2];
            spring_f32_pair<3>(d, o3, splat(A.oo2[sh]), make_float4(ti.k.hi, ti.r0.hi, ti.rc2.hi, ti.cor.hi),
                               make_float4(to.k.hi, to.r0.hi, to.rc2.hi, to.cor.hi), live, A.p24, A.p0, ff3, brk);
#pragma unroll
            for (int c = 0; c < 3; c++) {  // in the form of a split force
                f[c][0] = ff{-ff3[c][0], 0.0f};
                f[c][1] = ff{-ff3[c][1], 0.0f};
            }
        }
        if (brk[1]) newb |= (uint16_t)(1u << s);
        if (big) {
#pragma unroll
            for (int c = 0; c < 3; c++) {
                F[c].sub(f[c][0]);
                F[c].add(f[c][1]);
            }
        } else {
#pragma unroll
            for (int c = 0; c < 3; c++) {
                F[c].DfSum::sub(f[c][0]);
                F[c].DfSum::add(f[c][1]);
            }
        }
    }
}

// RATE: constant strain-rate loading (a separate instance, so that the
// ordinary step carries none of its code)
template <int PREC, int MODE, bool SAMPLE, bool RATE>
__global__ void __launch_bounds__(T3N, T3MIN)
k_tile3d(Tile3Args A)
{
    extern __shared__ __align__(16) unsigned char smem3[];
    Smem3 &S = *reinterpret_cast<Smem3 *>(smem3);
    __shared__ TypeDF sdf[128];
    __shared__ Coef4 scoef[8];
    __shared__ float smassf[8];
    __shared__ int soff[9];
    __shared__ int wcount[T3V / 32];  // particles per 32 voxels in block order, then the offsets
    __shared__ int ntotal;
    __shared__ double sred[T3N / 32];

    const int tid = threadIdx.x, lane = tid & 31;
    const int x0 = blockIdx.x * T3X, y0 = blockIdx.y * T3Y, z0 = blockIdx.z * T3Z;
    const int64_t tile_id = blockIdx.x + (int64_t)gridDim.x * (blockIdx.y + (int64_t)gridDim.y * blockIdx.z);
    const int nt = 2 * A.nphase * A.nphase;
    for (int q = tid; q < nt; q += T3N) sdf[q] = A.tdf[q];
    if (tid < A.nphase) {
        smassf[tid] = (float)A.mass[tid];
        scoef[tid] = A.coef[tid];
    }
    if (tid < 9) soff[tid] = A.sd[tid][0] + R3X * (A.sd[tid][1] + R3Y * A.sd[tid][2]);
    const long long step_now = MODE == T_STEP ? *A.d_step + A.t_off : 0;

    // 1. region (block + one-voxel halo) into shared memory
    bool over = false, bad = false;
    double rate_l = 0.0, rate_r = 0.0;  // grips' x under the constant strain rate
    if constexpr (RATE && MODE == T_STEP) {
        rate_l = rate_grip_x(A, 0);
        rate_r = rate_grip_x(A, A.nx - 1);
    }
    // the phases of all of a thread's voxels first, so that the loads that
    // depend on them wait once
    constexpr int KL = (R3N + T3N - 1) / T3N;
    RawVoxel raw[KL];
#pragma unroll
    for (int k = 0; k < KL; k++) {
        const int e = tid + k * T3N;
        raw[k] = e < R3N ? voxel_at(A, x0, y0, z0, e) : RawVoxel{-1, 0};
    }
#pragma unroll
    for (int k = 0; k < KL; k++) {
        const int e = tid + k * T3N;
        if (e < R3N) load_voxel<MODE, SAMPLE, RATE>(A, x0, e, raw[k], S, over, bad, rate_l, rate_r);
    }
    if (over) atomicOr(A.status, 2);
    __syncthreads();

    // 2. compact the block's particles (rows of 32 voxels; deterministic order:
    // raster order of the block) so that every warp works on particles
    for (int r = tid >> 5; r < T3V / 32; r += T3N / 32) {
        const int l = r * 32 + lane, lx = l % T3X, ly = (l / T3X) % T3Y, lz = l / (T3X * T3Y);
        const int ep = (lx + 1) + R3X * ((ly + 1) + R3Y * (lz + 1));
        const bool live = x0 + lx < A.nx && y0 + ly < A.ny && z0 + lz < A.nz && S.ph[ep];
        const unsigned b = __ballot_sync(0xffffffffu, live);
        if (lane == 0) wcount[r] = __popc(b);
    }
    __syncthreads();
    static_assert(T3V / 32 == 32, "one scan of 32 rows");
    if (tid < 32) {
        const int cnt = wcount[lane];
        int sum = cnt;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int u = __shfl_up_sync(0xffffffffu, sum, o);
            if (lane >= o) sum += u;
        }
        wcount[lane] = sum - cnt;
        if (lane == 31) ntotal = sum;
    }
    __syncthreads();
    for (int r = tid >> 5; r < T3V / 32; r += T3N / 32) {
        const int l = r * 32 + lane, lx = l % T3X, ly = (l / T3X) % T3Y, lz = l / (T3X * T3Y);
        const int ep = (lx + 1) + R3X * ((ly + 1) + R3Y * (lz + 1));
        const bool live = x0 + lx < A.nx && y0 + ly < A.ny && z0 + lz < A.nz && S.ph[ep];
        const unsigned b = __ballot_sync(0xffffffffu, live);
        if (live) S.list[wcount[r] + __popc(b & ((1u << lane) - 1u))] = (uint16_t)ep;
    }
    __syncthreads();

    // 3. each particle's 18 springs in canonical order, then the integration
    ff w_acc{0.0f, 0.0f}, u_acc{0.0f, 0.0f};
    float mvx2f = 0.0f, kef = 0.0f, resf = 0.0f;
    ff reactf{0.0f, 0.0f};
    const int count = ntotal;
    for (int i = tid; i < count; i += T3N) {
        const int ep = S.list[i];
        const int rx = ep % R3X, ry = (ep / R3X) % R3Y, rz = ep / (R3X * R3Y);
        const int gx = x0 + rx - 1, gy = y0 + ry - 1, gz = z0 + rz - 1;
        const int64_t g = gx + (int64_t)A.nx * (gy + (int64_t)A.ny * gz);
        const int pp = S.ph[ep];
        const uint16_t mk = S.mk[ep];
        const long long xp[3] = {S.xf[0][ep], S.xf[1][ep], S.xf[2][ep]};
        // time steps without a sample issue the integration's global loads
        // here, so their latency hides behind the springs (the sample
        // instance keeps them late: it has no registers to spare)
        constexpr bool PRE = MODE == T_STEP && !SAMPLE;
        double vpre[3];
        if constexpr (PRE) {
#pragma unroll
            for (int c = 0; c < 3; c++) vpre[c] = A.vh_in[c * A.nv + g];
        }
        // one spring at a time (sample steps), and in F32, whose forces are
        // plain floats (hi alone), the sums keep their errors
        DfSumCareful F3[3];
#pragma unroll
        for (int c = 0; c < 3; c++) F3[c].hs = F3[c].el = 0.0f;
        uint16_t newb = 0;
        if constexpr (MODE == T_STEP && !SAMPLE) {
            // a slot's incoming (source p - o_s) and outgoing (target p + o_s)
            // springs side by side on packed instructions
            tile3_pairs<PREC>(A, S, sdf, soff, ep, pp, mk, xp, F3, newb);
        } else {
            // the same springs in the same order, one at a time (initial accelerations
            // too, which have no break test: the pairs' springs beyond their critical
            // length give no force)
#pragma unroll 1
            for (int s = 0; s < 9; s++) {
                const int sh = A.ssh[s] - 1, ei = ep - soff[s], eo = ep + soff[s];
                const int pi = S.ph[ei], po = S.ph[eo];
                if (pi && !((S.mk[ei] >> s) & 1)) {
                    const long long xq[3] = {S.xf[0][ei], S.xf[1][ei], S.xf[2][ei]};
                    const TypeDF t = sdf[(((pi - 1) * A.nphase) + (pp - 1)) * 2 + sh];
                    ff f[3], wd{0.0f, 0.0f}, ud{0.0f, 0.0f};
                    if (spring3<PREC, MODE == T_STEP>(A, xq, xp, s, t, f, wd, ud, false)) {
#pragma unroll
                        for (int c = 0; c < 3; c++) F3[c].sub(f[c]);
                    }
                }
                if (po && !((mk >> s) & 1)) {
                    const long long xq[3] = {S.xf[0][eo], S.xf[1][eo], S.xf[2][eo]};
                    const TypeDF t = sdf[(((pp - 1) * A.nphase) + (po - 1)) * 2 + sh];
                    ff f[3];
                    if (spring3<PREC, MODE == T_STEP>(A, xp, xq, s, t, f, w_acc, u_acc, SAMPLE)) {
#pragma unroll
                        for (int c = 0; c < 3; c++) F3[c].add(f[c]);
                    } else {
                        newb |= (uint16_t)(1u << s);
                    }
                }
            }
        }
        if (MODE == T_STEP && newb) {
            for (int s = 0; s < 9; s++)
                if ((newb >> s) & 1) {
                    A.brk[(int64_t)s * A.nv + g] = step_now;
                    atomicMin(A.first_break, (unsigned long long)step_now);
                    atomicAdd(A.nbroken, 1ull);
                }
        }
        if (MODE == T_STEP && newb) A.mask[g] = (uint16_t)(mk | newb);

        // integration (Eqs. 4-5), FP64
        const bool grip = gx == 0 || gx == A.nx - 1;
        const int ph = pp - 1;
        if (SAMPLE && gx == A.nx - 1) reactf = ff_add_sloppy(reactf, ff{-F3[0].hs, -F3[0].el});
#pragma unroll
        for (int c = 0; c < 3; c++) {
            const bool fixed = grip && (c == 0 || A.grip_mode == 1);
            const int64_t q = c * A.nv + g;
            const double F = F3[c].value(A.df_bias);
            float Ff = __fadd_rn(F3[c].hs, F3[c].el);
            if (PREC == LSM_PREC_DF) Ff = __fmul_rn(Ff, A.p24);  // back from units of 2^(24-S)
            double vh;
            if constexpr (PRE) vh = vpre[c];
            else vh = MODE == T_INIT ? A.v_obs[q] : A.vh_in[q];
            if (fixed) {
                if (MODE == T_STEP) A.vh_out[q] = 0.0;
                if (MODE == T_STEP && SAMPLE) A.v_obs[q] = 0.0;
                continue;
            }
            if (MODE == T_OBSERVE) {
                if (SAMPLE) {
                    const float vf = d2f_bits(A.v_obs[q]);
                    resf = fmaxf(resf, fmaxf(fabsf(Ff), fabsf(vf)));
                    kef = fmaf(0.5f * smassf[ph] * vf, vf, kef);
                    if (c == 0) mvx2f = fmaf(smassf[ph] * vf, vf, mvx2f);
                }
                continue;
            }
            const Coef4 k4 = scoef[ph];
            const double vn = fma(k4.c2h, F, k4.c1h * vh);
            if (MODE == T_INIT) {
                A.vh_out[q] = vn;
                continue;
            }
            A.vh_out[q] = fma(k4.c2, F, k4.c1 * vh);
            if (SAMPLE) {
                A.v_obs[q] = vn;
                const float vf = d2f_bits(vn);
                resf = fmaxf(resf, fmaxf(fabsf(Ff), fabsf(vf)));
                kef = fmaf(0.5f * smassf[ph] * vf, vf, kef);
                if (c == 0) mvx2f = fmaf(smassf[ph] * vf, vf, mvx2f);
                bad |= !dbl_finite_bits(vn);
            }
        }
    }
    if (SAMPLE) {
        if (bad) atomicOr(A.status, 1);
        const double t0 = bsum_ff<T3N / 32>(w_acc, sred);
        const double t1 = bsum_ff<T3N / 32>(u_acc, sred);
        const double t2 = bsum_ff<T3N / 32>(ff{mvx2f, 0.0f}, sred);
        const double t3 = bsum_ff<T3N / 32>(ff{kef, 0.0f}, sred);
        const double t4 = bsum_ff<T3N / 32>(reactf, sred);
        const double t5 = bmax_f<T3N / 32>(resf, sred);
        if (tid == 0) {
            const double u = PREC == LSM_PREC_DF ? (double)A.p24 : 1.0;  // from units of 2^(24-S) (exact)
            A.part_s[tile_id] = t0 * (u * u);
            A.part_s[A.ntiles + tile_id] = t1 * (u * u);
            A.part_p[tile_id] = t2;
            A.part_p[A.ntiles + tile_id] = t3;
            A.part_p[2 * A.ntiles + tile_id] = t4 * u;
            A.part_p[3 * A.ntiles + tile_id] = t5;
        }
    }
}

// voxel-grid broken flags / break steps -> canonical spring order
__global__ void k_tile3_export(int nx, int ny, int nz, int64_t nv, Tile3Args A, const uint8_t *__restrict__ phase,
                               const uint16_t *__restrict__ mask, const long long *__restrict__ brk,
                               const int64_t *__restrict__ sbase, uint8_t *__restrict__ out_mask,
                               long long *__restrict__ out_brk)
{
    const int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (g >= nv || !phase[g]) return;
    const int gx = (int)(g % nx), gy = (int)((g / nx) % ny), gz = (int)(g / ((int64_t)nx * ny));
    int64_t b = sbase[g];
    const uint16_t mk = mask[g];
    for (int s = 0; s < 9; s++) {
        const int qx = gx + A.sd[s][0], qy = gy + A.sd[s][1], qz = gz + A.sd[s][2];
        if (qx < 0 || qx >= nx || qy < 0 || qy >= ny || qz < 0 || qz >= nz) continue;
        if (!phase[qx + (int64_t)nx * (qy + (int64_t)ny * qz)]) continue;
        if (out_mask) out_mask[b] = (mk >> s) & 1u;
        if (out_brk) out_brk[b] = brk[(int64_t)s * nv + g];
        b++;
    }
}

Tile3Args tile3_args(Ctx &c)
{
    Tile3Args A{};
    A.nx = c.h.nx;
    A.ny = c.h.ny;
    A.nz = c.h.nz;
    A.nphase = c.tile_nphase;
    A.nv = c.tnp;
    A.x_in = c.tx[c.tcur];
    A.vh_in = c.tvh[c.tcur];
    A.x_out = c.tx[c.tcur ^ 1];
    A.vh_out = c.tvh[c.tcur ^ 1];
    A.v_obs = c.tvobs;
    A.phase = c.tph;
    A.mask = c.tmask3;
    A.brk = c.tbrk;
    A.tdf = c.tdf;
    A.mass = c.tmass;
    A.coef = (const Coef4 *)c.tinvm;
    A.S = c.fix_S;
    A.a_fix = c.a_fix;
    A.p24 = ldexpf(1.0f, 24 - c.fix_S);
    A.p0 = ldexpf(1.0f, -c.fix_S);
    A.dt = c.h.dt;
    A.a = c.h.a;
    A.xc = c.h.xc;
    A.grip_mode = c.h.grip_mode;
    A.rate_on = c.rate_on;
    A.rate_eps0 = c.rate_eps0;
    A.rate_dt = c.rate_dt;
    A.rate_step0 = c.rate_step0;
    A.d_step = c.d_step;
    A.first_break = c.d_first_break;
    A.nbroken = c.d_nbroken;
    A.status = c.d_status;
    A.part_s = c.part_s;
    A.part_p = c.part_p;
    A.ntiles = c.ntiles;
    const double aa = std::ldexp((double)c.a_fix, -c.fix_S);
    for (int s = 0; s < 9; s++) {
        int l2 = 0;
        for (int k = 0; k < 3; k++) {
            A.sd[s][k] = (int)std::lround(c.h.offv[3 * s + k] / c.h.a);
            l2 += A.sd[s][k] * A.sd[s][k];
        }
        A.ssh[s] = l2;
    }
    A.fa = (float)aa;
    A.df_bias = (unsigned)(896 + (c.h.precision == LSM_PREC_DF ? 24 - c.fix_S : 0)) << 20;
    A.df_M = (float)std::ldexp(1.5 * c.df.unit, 23 + c.fix_S - 24);
    A.df_cmax = (float)c.df.cmax;
    A.oo2[0] = (float)(aa * aa);
    A.oo2[1] = (float)(2.0 * aa * aa);
    return A;
}

template <int PREC, int MODE, bool SAMPLE, bool RATE>
cudaError_t launch3(Ctx &c, Tile3Args A)
{
    auto kern = k_tile3d<PREC, MODE, SAMPLE, RATE>;
    static bool configured = false;  // per template instance
    if (!configured) {
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(Smem3));
        if (e == cudaSuccess) e = cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
        if (e != cudaSuccess) return e;
        configured = true;
    }
    const dim3 grid((c.h.nx + T3X - 1) / T3X, (c.h.ny + T3Y - 1) / T3Y, (c.h.nz + T3Z - 1) / T3Z);
    kern<<<grid, T3N, sizeof(Smem3), c.stream>>>(A);
    return cudaSuccess;
}

template <int MODE, bool SAMPLE>
cudaError_t launch3_prec(Ctx &c, Tile3Args A)
{
    if constexpr (MODE == T_STEP) {
        if (c.rate_on) {
            if (c.h.precision == LSM_PREC_F32) return launch3<LSM_PREC_F32, MODE, SAMPLE, true>(c, A);
            return launch3<LSM_PREC_DF, MODE, SAMPLE, true>(c, A);
        }
    }
    if (c.h.precision == LSM_PREC_F32) return launch3<LSM_PREC_F32, MODE, SAMPLE, false>(c, A);
    return launch3<LSM_PREC_DF, MODE, SAMPLE, false>(c, A);
}

ff split_ff3(double v)
{
    const float hi = (float)v;
    return ff{hi, (float)(v - (double)hi)};
}

template <typename T>
cudaError_t dal(T **p, size_t count)
{
    return lsm::dev_malloc((void **)p, (count ? count : 1) * sizeof(T));
}

}  // namespace

int64_t tile3_count(const Ctx &c)
{
    return (int64_t)((c.h.nx + T3X - 1) / T3X) * ((c.h.ny + T3Y - 1) / T3Y) * ((c.h.nz + T3Z - 1) / T3Z);
}

cudaError_t tile3_upload(Ctx &c)
{
    const HostNet &h = c.h;
    const int64_t nv = (int64_t)h.nx * h.ny * h.nz;
    c.tnp = nv;
    c.tile_nphase = h.nphase;
    c.ntiles = tile3_count(c);
    c.tgidx.assign(h.pix.begin(), h.pix.end());  // grid index of each particle: its voxel
    c.tgnx = h.nx;                                // rows of nx voxels, x fastest (the load
    c.tgny = h.ny * h.nz;                         // increment's kernel works per row)
    std::vector<double> X(3 * nv);
    for (int64_t g = 0; g < nv; g++) {
        X[g] = (g % h.nx) * h.a;
        X[nv + g] = ((g / h.nx) % h.ny) * h.a;
        X[2 * nv + g] = (g / ((int64_t)h.nx * h.ny)) * h.a;
    }
    std::vector<double> mtab(h.nphase, 1.0), itab(4 * h.nphase, 0.0);
    for (int64_t p = 0; p < h.n; p++) mtab[h.phase[h.pix[p]] - 1] = h.mass[p];
    for (int q = 0; q < h.nphase; q++) {
        const double dt = h.dt, hdt = 0.5 * h.dt, gm = h.damping, m = mtab[q];
        itab[4 * q + 0] = 1.0 - dt * gm / m;
        itab[4 * q + 1] = dt / m;
        itab[4 * q + 2] = 1.0 - hdt * gm / m;
        itab[4 * q + 3] = hdt / m;
    }
    const int maxext = std::max(h.nx, std::max(h.ny, h.nz));
    c.fix_S = 61 - (int)std::ceil(std::log2(4.0 * maxext * h.a + 16.0));
    c.fix_S = std::min(c.fix_S, 47 - (int)std::ceil(std::log2(h.a * std::sqrt(2.0))));
    c.fix_S = std::min(c.fix_S, 47 - (int)std::floor(std::log2(max_critical_length(h.types))));
    c.a_fix = std::llround(std::ldexp(h.a, c.fix_S));
    c.df = df_split(h.types, 6, 12);
    const double aa = std::ldexp((double)c.a_fix, -c.fix_S);
    std::vector<TypeDF> tdf(h.types.size());
    for (size_t q = 0; q < h.types.size(); q++) {
        const SpringType &t = h.types[q];
        const double shell = (q & 1) ? 2.0 : 1.0;
        const double p = t.r0 * t.r0, pe = std::fma(t.r0, t.r0, -p);
        const double o2 = shell * aa * aa, o2e = shell * std::fma(aa, aa, -(aa * aa));
        // DF: lengths in units of 2^(24-S) (exact power-of-two scaling)
        const double ul = h.precision == LSM_PREC_DF ? std::ldexp(1.0, c.fix_S - 24) : 1.0;
        tdf[q].k = split_ff3(t.k);
        tdf[q].r0 = split_ff3(t.r0 * ul);
        tdf[q].rc2 = split_ff3(t.rc2 * ul * ul);
        tdf[q].cor = split_ff3((o2 - p) + (o2e - pe));
    }
    std::vector<int64_t> sbase(nv, 0);
    for (int64_t s = h.m - 1; s >= 0; s--) sbase[h.pix[h.si[s]]] = s;
    cudaError_t e;
#define T3_TRY(x)                             \
    do {                                      \
        if ((e = (x)) != cudaSuccess) return e; \
    } while (0)
    for (int b = 0; b < 2; b++) {
        T3_TRY(dal(&c.tx[b], 3 * nv));
        T3_TRY(dal(&c.tvh[b], 3 * nv));
    }
    T3_TRY(dal(&c.tvobs, 3 * nv));
    T3_TRY(dal(&c.tph, nv));
    T3_TRY(dal(&c.tmask3, nv));
    T3_TRY(dal(&c.tbrk, 9 * nv));
    T3_TRY(dal(&c.tmass, h.nphase));
    T3_TRY(dal(&c.tinvm, 4 * h.nphase));
    T3_TRY(dal(&c.tdf, tdf.size()));
    T3_TRY(dal(&c.tsbase, nv));
    T3_TRY(dal(&c.part_s, 2 * c.ntiles));
    T3_TRY(dal(&c.part_p, 4 * c.ntiles));
    cudaStream_t st = c.stream;
    for (int b = 0; b < 2; b++) {
        T3_TRY(cudaMemcpyAsync(c.tx[b], X.data(), 3 * nv * sizeof(double), cudaMemcpyHostToDevice, st));
        T3_TRY(cudaMemsetAsync(c.tvh[b], 0, 3 * nv * sizeof(double), st));
    }
    T3_TRY(cudaMemsetAsync(c.tvobs, 0, 3 * nv * sizeof(double), st));
    T3_TRY(cudaMemcpyAsync(c.tph, h.phase.data(), nv, cudaMemcpyHostToDevice, st));
    T3_TRY(cudaMemsetAsync(c.tmask3, 0, nv * sizeof(uint16_t), st));
    T3_TRY(cudaMemsetAsync(c.tbrk, 0xff, 9 * nv * sizeof(long long), st));
    T3_TRY(cudaMemcpyAsync(c.tmass, mtab.data(), h.nphase * sizeof(double), cudaMemcpyHostToDevice, st));
    T3_TRY(cudaMemcpyAsync(c.tinvm, itab.data(), 4 * h.nphase * sizeof(double), cudaMemcpyHostToDevice, st));
    T3_TRY(cudaMemcpyAsync(c.tdf, tdf.data(), tdf.size() * sizeof(TypeDF), cudaMemcpyHostToDevice, st));
    T3_TRY(cudaMemcpyAsync(c.tsbase, sbase.data(), nv * sizeof(int64_t), cudaMemcpyHostToDevice, st));
    c.tcur = 0;
    T3_TRY(cudaStreamSynchronize(st));
#undef T3_TRY
    return cudaSuccess;
}

cudaError_t tile3_enqueue_steps(Ctx &c, int64_t nsteps, int start_buf, int &end_buf)
{
    int cur = start_buf;
    for (int64_t t = 0; t < nsteps; t++) {
        Tile3Args A = tile3_args(c);
        A.t_off = t;
        A.x_in = c.tx[cur];
        A.vh_in = c.tvh[cur];
        A.x_out = c.tx[cur ^ 1];
        A.vh_out = c.tvh[cur ^ 1];
        cudaError_t e = t == nsteps - 1 ? launch3_prec<T_STEP, true>(c, A) : launch3_prec<T_STEP, false>(c, A);
        if (e != cudaSuccess) return e;
        cur ^= 1;
    }
    end_buf = cur;
    return cudaGetLastError();
}

cudaError_t tile3_init_accel(Ctx &c)
{
    Tile3Args A = tile3_args(c);
    A.vh_out = c.tvh[c.tcur];
    cudaError_t e = launch3_prec<T_INIT, false>(c, A);
    if (e != cudaSuccess) return e;
    return cudaGetLastError();
}

cudaError_t tile3_observe(Ctx &c)
{
    cudaError_t e = launch3_prec<T_OBSERVE, true>(c, tile3_args(c));
    if (e != cudaSuccess) return e;
    return cudaGetLastError();
}

cudaError_t tile3_export(Ctx &c, bool steps)
{
    if (c.m == 0) return cudaSuccess;
    if (!c.texport) {
        cudaError_t e = lsm::dev_malloc((void **)&c.texport, c.m);
        if (e != cudaSuccess) return e;
    }
    if (steps && !c.texport_brk) {
        cudaError_t e = lsm::dev_malloc((void **)&c.texport_brk, c.m * sizeof(long long));
        if (e != cudaSuccess) return e;
    }
    const unsigned g = (unsigned)((c.tnp + 255) / 256);
    k_tile3_export<<<g, 256, 0, c.stream>>>(c.h.nx, c.h.ny, c.h.nz, c.tnp, tile3_args(c), c.tph, c.tmask3, c.tbrk,
                                            c.tsbase, steps ? nullptr : c.texport,
                                            steps ? c.texport_brk : nullptr);
    return cudaGetLastError();
}

}  // namespace lsm
