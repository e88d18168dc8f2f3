// k_march2 for FP32 storage with the cascaded scalar model.
#include "ddflb_march.cuh"

namespace ddflb {
cudaError_t launch_march2_cascaded(const Launch& L, const void* fin, const void* gin, void* fout,
                                   void* gout, DevStatus* st, int rows) {
  return L.force ? march::go_bc<float, true, 2>(L, fin, gin, fout, gout, st, rows)
                 : march::go_bc<float, false, 2>(L, fin, gin, fout, gout, st, rows);
}
}  // namespace ddflb
