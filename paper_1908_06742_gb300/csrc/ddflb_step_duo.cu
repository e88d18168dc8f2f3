// One time step with two adjacent nodes per thread and packed FP32 arithmetic
// (k_step_duo), for the unforced MRT and SRT lattices between those that take
// four steps per launch and those that take two (which kernel where:
// ddflb_api.cu).
#include <cuda_runtime.h>

#include "ddflb_device.cuh"
#include "ddflb_internal.h"
#include "ddflb_pair.cuh"

namespace ddflb {

template <typename S>
struct DuoIo {  // 16-bit storage: the pair is one 4-byte word
  static __device__ __forceinline__ F2 ldg(const S* p) {
    return widen<S>(__ldg(reinterpret_cast<const unsigned*>(p)));
  }
  static __device__ __forceinline__ float ldg1(const S* p) { return widen1(__ldg(p)); }
  static __device__ __forceinline__ void st(S* p, F2 v) {
    *reinterpret_cast<unsigned*>(p) = narrow<S>(v);
  }
};
template <>
struct DuoIo<float> {
  static __device__ __forceinline__ F2 ldg(const float* p) {
    return __ldg(reinterpret_cast<const float2*>(p));
  }
  static __device__ __forceinline__ float ldg1(const float* p) { return __ldg(p); }
  static __device__ __forceinline__ void st(float* p, F2 v) { *reinterpret_cast<float2*>(p) = v; }
};

// Lattices of this size sit in L2 or straddle it, so the step is bound by issue
// and by L2, not by the copy bandwidth.  A pair shares its arithmetic's issue
// slots (ddflb_pair.cuh) and its addresses; the stores keep their lines in L2 for
// the next step.  down: the rows in descending order; taken every other step
// where the two buffers exceed L2, so that a step begins with the rows the last
// one ended with.  us per step, one node per thread -> this: FP32 512^2 5.96 ->
// 5.36, 700^2 10.1 -> 8.4, 1024^2 24.5 -> 20.4 (22.2 without alternating); FP16
// 1023^2 16.3 -> 12.0; 16-bit cavities (from the four-node kernel, whose groups
// next to a wall go node by node) 700^2 13.1 -> 7.6, 1024^2 19.6 -> 13.2, 2048^2
// 64.9 -> 56.1.  Below about 450^2 FP32 the one-node kernel has more warps to hide
// latency with and stays (384^2: 4.07 against 4.39).  4 or 6 CTAs per SM: 24.2 and
// 25.0 at 1024^2 (5: 22.9), evict-first stores 21.2.
template <typename S, int BC>
__global__ void __launch_bounds__(128, 5)
    k_step_duo(LbParams P, PairConst K, const S* __restrict__ fin, const S* __restrict__ gin,
               S* __restrict__ fout, S* __restrict__ gout, const DevStatus* __restrict__ status,
               bool down) {
  using Io = DuoIo<S>;
  constexpr bool COMP = sizeof(S) == 4;
  const int nx = P.nx, ny = P.ny;
  const int x0 = 2 * (blockIdx.x * 128 + threadIdx.x);
  const int y = down ? ny - 1 - (int)blockIdx.y : (int)blockIdx.y;
  if (x0 >= nx || status->diverged) return;
  F2 df[9], dg[9];
  if (BC == BC_PERIODIC || (y >= 1 && y < ny - 1)) {
    const int ym = y == 0 ? ny - 1 : y - 1, yp = y == ny - 1 ? 0 : y + 1;
    // columns the first node pulls from on its left, the two nodes on their
    // right (wrapped; a cavity's links beyond its walls are replaced below)
    const int xm = x0 == 0 ? nx - 1 : x0 - 1;
    const int xa = x0 + 1 >= nx ? 0 : x0 + 1, xb = x0 + 2 >= nx ? max(x0 + 2 - nx, 0) : x0 + 2;
    const uint32_t ro[3] = {(uint32_t)ym * (uint32_t)P.pitch, (uint32_t)y * (uint32_t)P.pitch,
                            (uint32_t)yp * (uint32_t)P.pitch};
#pragma unroll
    for (int a = 0; a < 9; ++a) {
      constexpr int EX[9] = {0, 1, 0, -1, 0, 1, -1, -1, 1};
      constexpr int EY[9] = {0, 0, 1, 0, -1, 1, 1, -1, -1};
      const S* const f = fin + a * P.plane + ro[1 - EY[a]];
      const S* const g = gin + a * P.plane + ro[1 - EY[a]];
      if (EX[a] == 0) {
        df[a] = Io::ldg(f + x0);
        dg[a] = Io::ldg(g + x0);
      } else {
        const int u = EX[a] == 1 ? xm : xa, v = EX[a] == 1 ? x0 : min(xb, nx - 1);
        df[a] = make_float2(Io::ldg1(f + u), Io::ldg1(f + v));
        dg[a] = make_float2(Io::ldg1(g + u), Io::ldg1(g + v));
      }
    }
    if (BC == BC_CAVITY && (x0 == 0 || x0 + 2 >= nx)) {
      // links beyond a side wall: the own value of the opposite direction (pull())
      const uint32_t own = ro[1];
      auto bounce = [&](int a, int b, int x, float& vf, float& vg) {
        vf = Codec<S>::load(fin + b * P.plane + own + x, P.isf) + 0.0f;
        vg = P.abb_wall[a] - Codec<S>::load(gin + b * P.plane + own + x, P.isg);
        if (!COMP) {  // in storage units (a power of two: exact)
          vf *= P.sf;
          vg *= P.sg;
        }
      };
      if (x0 == 0) {
        bounce(1, 3, 0, df[1].x, dg[1].x);
        bounce(5, 7, 0, df[5].x, dg[5].x);
        bounce(8, 6, 0, df[8].x, dg[8].x);
      }
      if (x0 == nx - 1) {
        bounce(3, 1, x0, df[3].x, dg[3].x);
        bounce(6, 8, x0, df[6].x, dg[6].x);
        bounce(7, 5, x0, df[7].x, dg[7].x);
      } else if (x0 + 1 == nx - 1) {
        bounce(3, 1, x0 + 1, df[3].y, dg[3].y);
        bounce(6, 8, x0 + 1, df[6].y, dg[6].y);
        bounce(7, 5, x0 + 1, df[7].y, dg[7].y);
      }
    }
  } else {
    // a row next to a wall: node by node
#pragma unroll 1
    for (int k = 0; k < 2; ++k) {
      float vf[9], vg[9];
      pull<S, BC>(P, fin, gin, min(x0 + k, nx - 1), y, vf, vg);
#pragma unroll
      for (int a = 0; a < 9; ++a) {
        const float f = COMP ? vf[a] : vf[a] * P.sf, g = COMP ? vg[a] : vg[a] * P.sg;
        if (k) df[a].y = f, dg[a].y = g;
        else df[a].x = f, dg[a].x = g;
      }
    }
  }
  collide_pair<COMP>(K, df, dg);
  // (where nx is odd the last pair's second value lands in the row's padding)
  const int64_t o = (int64_t)y * P.pitch + x0;
#pragma unroll
  for (int a = 0; a < 9; ++a) {
    Io::st(fout + a * P.plane + o, df[a]);
    Io::st(gout + a * P.plane + o, dg[a]);
  }
}

namespace {
template <typename S, int BC>
cudaError_t go(const Launch& L, const void* fin, const void* gin, void* fout, void* gout,
                    const DevStatus* st, bool down) {
  const dim3 g((L.P.nx + 255) / 256, L.P.ny);
  k_step_duo<S, BC><<<g, 128, 0, L.stream>>>(L.P, make_pair_const(L.P), (const S*)fin, (const S*)gin,
                                             (S*)fout, (S*)gout, st, down);
  return cudaGetLastError();
}
template <typename S>
cudaError_t go_bc(const Launch& L, const void* fin, const void* gin, void* fout, void* gout,
                  const DevStatus* st, bool down) {
  switch (L.P_bc) {
    case BC_PERIODIC: return go<S, BC_PERIODIC>(L, fin, gin, fout, gout, st, down);
    case BC_CAVITY: return go<S, BC_CAVITY>(L, fin, gin, fout, gout, st, down);
    default: return go<S, BC_CHANNEL>(L, fin, gin, fout, gout, st, down);
  }
}
}  // namespace

cudaError_t launch_step_duo(const Launch& L, const void* fin, const void* gin, void* fout,
                            void* gout, const DevStatus* st, bool down) {
  switch (L.storage) {
    case 0: return go_bc<float>(L, fin, gin, fout, gout, st, down);
    case 1: return go_bc<__half>(L, fin, gin, fout, gout, st, down);
    default: return go_bc<__nv_bfloat16>(L, fin, gin, fout, gout, st, down);
  }
}

}  // namespace ddflb
