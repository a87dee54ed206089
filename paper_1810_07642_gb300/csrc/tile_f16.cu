// Tile form of the step (tflbm_tile.cuh) with FP16 and BF16 populations.
#include "tflbm_tile.cuh"

namespace tflbm {

cudaError_t tile_step_narrow(int store, int block_x, const void* fin, void* fout, const void* kappa, void* mom, const Geom& G,
                             const Consts<float>& C, cudaStream_t st)
{
    if (store == kStoreF16) return tile_step<__half, float>(block_x, fin, fout, kappa, mom, G, C, st);
    if (store == kStoreBF16) return tile_step<__nv_bfloat16, float>(block_x, fin, fout, kappa, mom, G, C, st);
    return cudaErrorInvalidValue;
}

}  // namespace tflbm
