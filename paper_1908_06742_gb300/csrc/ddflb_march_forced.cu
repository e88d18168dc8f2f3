// k_march2 for FP32 storage with a uniform force.
#include "ddflb_march.cuh"

namespace ddflb {
cudaError_t launch_march2_forced(const Launch& L, const void* fin, const void* gin, void* fout,
                                 void* gout, DevStatus* st, int rows) {
  return march::go_bc<float, true, 0>(L, fin, gin, fout, gout, st, rows);
}
}  // namespace ddflb
