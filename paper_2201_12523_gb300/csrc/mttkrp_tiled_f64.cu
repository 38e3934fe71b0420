// Tile-order MTTKRP kernels with float64 values, factors and sums.
#include "mttkrp_tiled.cuh"

namespace blco {

cudaError_t launch_mttkrp_tiled_f64(const StoreView &sv, const TileOrder &to, const double *const *factors, int R,
                                    int mode, const HotRows &hot, double *out, cudaStream_t s) {
    if (sv.end <= 0) return cudaSuccess;
    TParams p = tiled_params(sv, to, reinterpret_cast<const void *const *>(factors), mode, hot, R * sizeof(double));
    p.vals_aligned = 1;
    p.out = out;
    switch (R) {
        case 8: return tiled64_by_ng<8>(p, s);
        case 16: return tiled64_by_ng<16>(p, s);
        case 32: return tiled64_by_ng<32>(p, s);
        case 64: return tiled64_by_ng<64>(p, s);
    }
    return cudaErrorInvalidValue;
}

}  // namespace blco
