// instantiates k_step_tile for F32 storage, with an obstacle mask
#include "lbm_step_tile.cuh"

namespace lbm {
cudaError_t step_tile_mask_f32(int coll, int K, const TileDom &d, const void *fin, void *fout, cudaStream_t s) {
    return TileDispatch<ST_F32, true>::step(coll, K, d, fin, fout, s);
}
}  // namespace lbm
