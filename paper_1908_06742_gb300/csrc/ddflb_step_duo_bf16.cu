// BF16 instances of the single-step kernel with two nodes per thread (ddflb_step_duo.cuh).
#include "ddflb_step_duo.cuh"

namespace ddflb {
cudaError_t launch_step_duo_bf16(const Launch& L, const void* fin, const void* gin, void* fout,
                                void* gout, const DevStatus* st, bool down) {
  return duo::go_bc<__nv_bfloat16>(L, fin, gin, fout, gout, st, down);
}
}  // namespace ddflb
