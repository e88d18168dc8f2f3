// k_march2 for __nv_bfloat16 storage (one translation unit per storage type).
#include "ddflb_march.cuh"

namespace ddflb {
cudaError_t launch_march2_bf16(const Launch& L, const void* fin, const void* gin, void* fout,
                           void* gout, DevStatus* st, int rows) {
  return march::go_bc<__nv_bfloat16, false, 0>(L, fin, gin, fout, gout, st, rows);
}
}  // namespace ddflb
