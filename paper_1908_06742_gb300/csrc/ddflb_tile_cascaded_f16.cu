// k_tile with the cascaded scalar model for __half storage (one translation unit per storage type).
#include "ddflb_tile.cuh"

namespace ddflb {
cudaError_t launch_tile_cascaded_f16(const Launch& L, const void* fin, const void* gin, void* fout,
                                     void* gout, const DevStatus* st, int shape) {
  return tile::go_bc<__half, 2>(L, fin, gin, fout, gout, st, shape);
}
}  // namespace ddflb
