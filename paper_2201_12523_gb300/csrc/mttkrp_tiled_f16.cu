// Tile-order MTTKRP kernels for __half factors.
#include "mttkrp_tiled.cuh"

namespace blco {

cudaError_t launch_mttkrp_tiled_f16(const StoreView &sv, const TileOrder &to, const FactorSet &fs, int R, int mode,
                                    const HotRows &hot, float *out, const OutCopies &oc, cudaStream_t s) {
    return tiled_as<__half>(sv, to, fs, R, mode, hot, out, oc, s);
}

}  // namespace blco
