// tile_multi.cu -- the multi-step tile kernel of small 2D images (tile_multi.cuh)
// and the rule that chooses it.
#include "tile_multi.cuh"

namespace lsm {

namespace {

template <int TX, int TY, int H, int G, int PREC, bool RATE, bool SAMPLE>
__global__ void __launch_bounds__((MultiShape<TX, TY, H, G>::NT))
k_tile_multi(TileArgs A, int ns)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    tile_multi_body<TX, TY, H, G, PREC, RATE, SAMPLE>(A, blockIdx.x, blockIdx.y,
                                                      (int64_t)blockIdx.y * gridDim.x + blockIdx.x, ns, smem_raw);
}

template <int TX, int TY, int H, int G, int PREC, bool RATE, bool SAMPLE>
cudaError_t launch_t(Ctx &c, TileArgs A, int ns)
{
    auto kern = k_tile_multi<TX, TY, H, G, PREC, RATE, SAMPLE>;
    constexpr size_t smem = multi_smem_bytes<TX, TY, H, G, PREC>();
    static bool configured = false;  // per template instance
    if (!configured) {
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e == cudaSuccess) e = cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
        if (e != cudaSuccess) return e;
        configured = true;
    }
    const dim3 grid((A.nx + TX - 1) / TX, (A.ny + TY - 1) / TY);
    A.ntiles = c.multi.tiles;  // partial-sum stride
    kern<<<grid, MultiShape<TX, TY, H, G>::NT, smem, c.stream>>>(A, ns);
    return cudaGetLastError();
}

template <int TX, int TY, int H, int G, int PREC>
cudaError_t launch_p(Ctx &c, const TileArgs &A, int ns, bool sample)
{
    if (c.rate_on)
        return sample ? launch_t<TX, TY, H, G, PREC, true, true>(c, A, ns)
                      : launch_t<TX, TY, H, G, PREC, true, false>(c, A, ns);
    return sample ? launch_t<TX, TY, H, G, PREC, false, true>(c, A, ns)
                  : launch_t<TX, TY, H, G, PREC, false, false>(c, A, ns);
}

bool exact_mode(int prec) { return prec == LSM_PREC_EXACT64 || prec == LSM_PREC_FAST64; }

}  // namespace

// Whether an nx x ny image runs on the multi-step kernel, and in which shape.
// Measured per time step in calls of 200, one-step tile kernel -> this one:
//   DF, F32: 16 x 4 tiles, halo 3, while they are at most about one per SM (64^2:
//   5.1 -> 1.9 us; 100 x 90: 5.5 -> 2.2); then 32 x 8 tiles, halo 2, up to two per SM
//   (200 x 150: 5.5 -> 3.0; 300 x 200: 6.3 -> 4.4; 400 x 400 would be even).
//   Exact: a spring's integer arithmetic is the chain (some 500 instructions)
//   and a halo's FP64 work costs more than a launch, so one step per launch with
//   four threads per cell, one spring each: 16 x 4 tiles up to one per two SMs
//   (64^2: 11.3 -> 6.4 us; a halo of 2 with two threads per cell 6.7), then 32 x 4
//   up to one per SM (100 x 90: 11.5 -> 8.6); 200 x 150 would lose (11.7, 16).
MultiPlan multi_shape(int prec, int nx, int ny, int sms)
{
    auto tiles = [&](int tx, int ty) { return (int64_t)((nx + tx - 1) / tx) * ((ny + ty - 1) / ty); };
    MultiPlan m;
    if (exact_mode(prec)) {
        if (tiles(16, 4) <= sms / 2) m = MultiPlan{MULTI_E16x4, 1, tiles(16, 4)};
        else if (tiles(32, 4) <= sms) m = MultiPlan{MULTI_E32x4, 1, tiles(32, 4)};
    } else {
        if (tiles(16, 4) <= sms + sms / 16) m = MultiPlan{MULTI_16x4, 3, tiles(16, 4)};
        else if (tiles(32, 8) <= 2 * sms) m = MultiPlan{MULTI_32x8, 2, tiles(32, 8)};
    }
    return m;
}

// ns (at most c.multi.halo) time steps in one launch.
cudaError_t launch_multi(Ctx &c, const TileArgs &A, int ns, bool sample)
{
    const bool df = c.h.precision == LSM_PREC_DF;
    switch (c.multi.shape) {
    case MULTI_16x4:
        return df ? launch_p<16, 4, 3, 1, LSM_PREC_DF>(c, A, ns, sample)
                  : launch_p<16, 4, 3, 1, LSM_PREC_F32>(c, A, ns, sample);
    case MULTI_32x8:
        return df ? launch_p<32, 8, 2, 1, LSM_PREC_DF>(c, A, ns, sample)
                  : launch_p<32, 8, 2, 1, LSM_PREC_F32>(c, A, ns, sample);
    case MULTI_E16x4: return launch_p<16, 4, 1, 4, LSM_PREC_EXACT64>(c, A, ns, sample);
    case MULTI_E32x4: return launch_p<32, 4, 1, 4, LSM_PREC_EXACT64>(c, A, ns, sample);
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace lsm
