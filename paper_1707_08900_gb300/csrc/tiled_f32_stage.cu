// The FP32 default kernel (tiled4_impl.cuh) on grids that are not whole tiles,
// with four fields or with unequal spacings: one instantiation per RK3 substep
// (substep 1 reads no u-tilde, substep 3 writes none), the grid-extent test kept.
// Whole tiles with five fields and equal spacing have their own instantiations
// beside the general one (tiled_f32.cu); forced steps and the other arithmetic
// forms take the substep at run time.
#include "tiled4_impl.cuh"

namespace gbfd {

namespace {

template <int NF, class CoefT, int STG>
cudaError_t launch(const StateBufs &b, const CoefT &c, const RKStage &st, int zc, int *dev_error,
                   const CUtensorMap &map, const CUtensorMap &wmap, cudaStream_t stream)
{
    constexpr int TX = 32, TY = 8, NS = 8, U = 2;
    constexpr auto kern = tiled4::k_substep_lag<float, float, NF, TX, TY, NS, U, 1, false, false, true,
                                                CoefT, false, STG, false>;
    const int tiles_x = (b.Ls.nx + TX - 1) / TX, tiles_y = (b.Ls.ny + TY - 1) / TY;
    return launch_chained<kern>(dim3(tiles_x * tiles_y, (b.Ls.nz + zc - 1) / zc), dim3(TX / 2 * TY),
                                tiled4::RingL<float, NF, TX, TY, NS, U>::BYTES, false, stream, map,
                                wmap, (float *)b.out, (float *)b.w, b.Ls, b.Lw, c, st, zc, tiles_x,
                                dev_error, st.fault_skip_plane);
}

template <int NF, class CoefT>
cudaError_t launch_s(const StateBufs &b, const CoefT &c, const RKStage &st, int zc, int *dev_error,
                     const CUtensorMap &map, const CUtensorMap &wmap, cudaStream_t stream)
{
    if (st.s == 0)
        return launch<NF, CoefT, 0>(b, c, st, zc, dev_error, map, wmap, stream);
    if (st.s == 1)
        return launch<NF, CoefT, 1>(b, c, st, zc, dev_error, map, wmap, stream);
    return launch<NF, CoefT, 2>(b, c, st, zc, dev_error, map, wmap, stream);
}

}  // namespace

cudaError_t launch_lag_stage(const StateBufs &b, const Coef<float> &c, const RKStage &st, int nf,
                             int zc, int cfg_key, int *dev_error, TmapCache *cache,
                             cudaStream_t stream, int *launches)
{
    CUtensorMap *map = nullptr, *wmap = nullptr;
    if (!get_state_tmap(cache, b.in, b.Ls, nf, 32, 8, cfg_key, &map) ||
        !get_tile_tmap(cache, b.w, b.Lw, nf, 32, 8, cfg_key, &wmap))
        return cudaErrorInvalidValue;
    const bool iso = coef_is_cubic(c);
    *launches += 1;
    if (nf == 5)
        return iso ? launch_s<5>(b, cubic_of(c), st, zc, dev_error, *map, *wmap, stream)
                   : launch_s<5>(b, c, st, zc, dev_error, *map, *wmap, stream);
    return iso ? launch_s<4>(b, cubic_of(c), st, zc, dev_error, *map, *wmap, stream)
               : launch_s<4>(b, c, st, zc, dev_error, *map, *wmap, stream);
}

}  // namespace gbfd
