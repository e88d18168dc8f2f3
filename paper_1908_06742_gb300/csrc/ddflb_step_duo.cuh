// One time step with two adjacent nodes per thread and packed FP32 arithmetic
// (k_step_duo), for the lattices between those that take four steps per launch
// and those that take two, and above the four-step kernel's at any size for what
// the two-step kernel does not serve: force fields, time-dependent forces, and
// 16-bit storage with a force or a central-moment scalar model (which kernel
// where: ddflb_api.cu).
#pragma once

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

// Most lattices here sit in L2 or straddle it, so the step is bound by issue and by
// L2, not by the copy bandwidth; with a force or a central-moment model the one-node
// kernel is bound by issue at every size (805 instructions a node, forced cascaded
// FP32).  A pair shares its arithmetic's issue slots (ddflb_pair.cuh) and its
// addresses; the stores keep their lines in L2 for the next step.  down: the rows in
// descending order; taken every other step where the two buffers exceed L2, so that
// a step begins with the rows the last one ended with.  us per step, one node per
// thread -> this:
//   MRT FP32              420^2 5.15 -> 4.21   701^2 10.2 -> 8.5   1024^2 24.4 -> 20.4
//   MRT BF16              420^2 4.62 -> 3.42   701^2 9.2 -> 6.6
//   forced cascaded FP32  701^2 13.3 -> 10.6   1024^2 29.8 -> 23.5   4096^2 425 -> 350
//   forced cascaded BF16  701^2 11.9 -> 9.1    1024^2 22.2 -> 17.2   4096^2 338 -> 258
// (1024^2 FP32 22.2 without alternating.)  16-bit cavities, from the four-node kernel,
// whose groups next to a wall go node by node: 1024^2 19.6 -> 13.2, 2048^2 64.9 ->
// 56.1.  Five CTAs per SM throughout: with four, forced cascaded BF16 4096^2 272
// (and MRT FP32 1024^2 24.2; six 25.0, evict-first stores 21.2 against 20.4).
template <typename S, int BC, bool FORCE, int SM, int BX>
__global__ void __launch_bounds__(128, 5)
    k_step_duo(LbParams P, PairConst K, const S* __restrict__ fin, const S* __restrict__ gin,
               S* __restrict__ fout, S* __restrict__ gout, const DevStatus* __restrict__ status,
               bool down) {
  using Io = DuoIo<S>;
  constexpr bool COMP = sizeof(S) == 4;
  // 16-bit populations stay in storage units where the collision allows it
  constexpr bool UNITS = !COMP && (FORCE || SM != 0);
  const int nx = P.nx, ny = P.ny;
  const int x0 = 2 * (blockIdx.x * (BX ? BX : blockDim.x) + threadIdx.x);
  const int y = down ? ny - 1 - (int)blockIdx.y : (int)blockIdx.y;
  if (x0 >= nx || status->stopped) return;
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
    if (UNITS) {
#pragma unroll
      for (int a = 0; a < 9; ++a) {
        df[a] = mul2(df[a], K.isf);
        dg[a] = mul2(dg[a], K.isg);
      }
    }
    if (BC == BC_CAVITY && (x0 == 0 || x0 + 2 >= nx)) {
      // links beyond a side wall: the own value of the opposite direction (pull())
      const uint32_t own = ro[1];
      auto bounce = [&](int a, int b, int x, float& vf, float& vg) {
        vf = Codec<S>::load(fin + b * P.plane + own + x, P.isf) + 0.0f;
        vg = P.abb_wall[a] - Codec<S>::load(gin + b * P.plane + own + x, P.isg);
        if (!COMP && !UNITS) {  // in storage units (a power of two: exact)
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
        const bool own = COMP || UNITS;
        const float f = own ? vf[a] : vf[a] * P.sf, g = own ? vg[a] : vg[a] * P.sg;
        if (k) df[a].y = f, dg[a].y = g;
        else df[a].x = f, dg[a].x = g;
      }
    }
  }
  F2 Fx{}, Fy{};
  if (FORCE) {
    const Force a = node_force(P, x0, y), b = node_force(P, min(x0 + 1, nx - 1), y);
    Fx = make_float2(a.x, b.x);
    Fy = make_float2(a.y, b.y);
  }
  collide_pair<COMP, FORCE, SM>(K, df, dg, Fx, Fy);
  // (where nx is odd the last pair's second value lands in the row's padding)
  const int64_t o = (int64_t)y * P.pitch + x0;
#pragma unroll
  for (int a = 0; a < 9; ++a) {
    Io::st(fout + a * P.plane + o, UNITS ? mul2(df[a], K.sf) : df[a]);
    Io::st(gout + a * P.plane + o, UNITS ? mul2(dg[a], K.sg) : dg[a]);
  }
}

namespace duo {
template <typename S, int BC, bool FORCE, int SM>
cudaError_t go(const Launch& L, const void* fin, const void* gin, void* fout, void* gout,
               const DevStatus* st, bool down) {
  // blocks of 128 pairs of one row, or of 64 or 32 where that leaves fewer threads
  // without a node (350^2: 6 blocks of 32 a row instead of 2 of 128); the widest as a
  // constant (1024^2 20.9 us per step with the width read at run time, 20.4 so)
  const int pairs = (L.P.nx + 1) / 2;
  int bx = 128;
  for (int b : {64, 32})
    if ((pairs + b - 1) / b * b < (pairs + bx - 1) / bx * bx) bx = b;
  const dim3 g((pairs + bx - 1) / bx, L.P.ny);
  auto* kernel = bx == 128 ? k_step_duo<S, BC, FORCE, SM, 128> : k_step_duo<S, BC, FORCE, SM, 0>;
  kernel<<<g, bx, 0, L.stream>>>(L.P, make_pair_const(L.P), (const S*)fin, (const S*)gin,
                                 (S*)fout, (S*)gout, st, down);
  return cudaGetLastError();
}
template <typename S, int BC, bool FORCE>
cudaError_t go_model(const Launch& L, const void* fin, const void* gin, void* fout, void* gout,
                     const DevStatus* st, bool down) {
  switch (L.P.smodel) {
    case 2: return go<S, BC, FORCE, 2>(L, fin, gin, fout, gout, st, down);
    case 3: return go<S, BC, FORCE, 3>(L, fin, gin, fout, gout, st, down);
    default: return go<S, BC, FORCE, 0>(L, fin, gin, fout, gout, st, down);
  }
}
template <typename S, int BC>
cudaError_t go_force(const Launch& L, const void* fin, const void* gin, void* fout, void* gout,
                     const DevStatus* st, bool down) {
  return L.force ? go_model<S, BC, true>(L, fin, gin, fout, gout, st, down)
                 : go_model<S, BC, false>(L, fin, gin, fout, gout, st, down);
}
template <typename S>
cudaError_t go_bc(const Launch& L, const void* fin, const void* gin, void* fout, void* gout,
                  const DevStatus* st, bool down) {
  switch (L.P_bc) {
    case BC_PERIODIC: return go_force<S, BC_PERIODIC>(L, fin, gin, fout, gout, st, down);
    case BC_CAVITY: return go_force<S, BC_CAVITY>(L, fin, gin, fout, gout, st, down);
    default: return go_force<S, BC_CHANNEL>(L, fin, gin, fout, gout, st, down);
  }
}
}  // namespace duo

}  // namespace ddflb
