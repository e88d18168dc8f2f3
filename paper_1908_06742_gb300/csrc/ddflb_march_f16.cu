// k_march2 for __half storage (one translation unit per storage type).
#include "ddflb_march.cuh"

namespace ddflb {
cudaError_t launch_march2_f16(const Launch& L, const void* fin, const void* gin, void* fout,
                           void* gout, DevStatus* st, int rows) {
  return march::go_bc<__half, false, 0>(L, fin, gin, fout, gout, st, rows);
}
}  // namespace ddflb
