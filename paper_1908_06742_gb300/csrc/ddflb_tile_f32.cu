// k_tile for float storage (one translation unit per storage type).
#include "ddflb_tile.cuh"

namespace ddflb {
cudaError_t launch_tile_f32(const Launch& L, const void* fin, const void* gin, void* fout,
                          void* gout, const DevStatus* st, int shape) {
  return tile::go_bc<float, 0>(L, fin, gin, fout, gout, st, shape);
}
}  // namespace ddflb
