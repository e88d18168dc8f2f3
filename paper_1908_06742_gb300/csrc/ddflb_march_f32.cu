// k_march2 for float storage (one translation unit per storage type).
#include "ddflb_march.cuh"

namespace ddflb {
cudaError_t launch_march2_f32(const Launch& L, const void* fin, const void* gin, void* fout,
                           void* gout, DevStatus* st, int rows) {
  return march::go_bc<float, false, 0>(L, fin, gin, fout, gout, st, rows);
}
}  // namespace ddflb
