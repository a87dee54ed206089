// Tile form of the step (tflbm_tile.cuh) with FP32 and FP64 populations.
#include "tflbm_tile.cuh"

namespace tflbm {

cudaError_t tile_step_narrow(int store, int block_x, const void* fin, void* fout, const void* kappa, void* mom, const Geom& G,
                             const Consts<float>& C, cudaStream_t st);

cudaError_t launch_tile(int store, int block_x, const void* fin, void* fout, const void* kappa, void* mom,
                        const Geom& G, const Consts<float>* C32, const Consts<double>* C64, cudaStream_t st)
{
    switch (store) {
        case kStoreF32: return tile_step<float, float>(block_x, fin, fout, kappa, mom, G, *C32, st);
        case kStoreF64: return tile_step<double, double>(block_x, fin, fout, kappa, mom, G, *C64, st);
        default: return tile_step_narrow(store, block_x, fin, fout, kappa, mom, G, *C32, st);
    }
}

}  // namespace tflbm
