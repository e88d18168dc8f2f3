// Several fused time steps per launch for small lattices (k_tile): see the
// kernel's comment.  Included by one translation unit per storage type.
#pragma once

#include <cuda_runtime.h>

#include "ddflb_device.cuh"
#include "ddflb_internal.h"
#include "ddflb_smem.h"

namespace ddflb {

// One CTA takes a tile of TX x TY nodes through T steps.  Level l = 1 .. T
// computes the state after l steps on the tile and T - l nodes around it, so
// that CTAs need nothing from each other within a launch; levels 1 .. T - 1
// stay in shared memory (two buffers, read and written in turn).
//
// A small lattice is bound by the launch and by the length of one thread's
// instruction stream (about 520 instructions a node and level; 64^2: five warps on
// the four schedulers at the first level), not by any rate; the largest tile, 32 x
// 14, has 24 to 14 warps a level and spends more than half of a launch on issue.
// One step per launch takes 2.0 us at 64^2 FP32, four per launch 0.90 us a step, the redundant nodes included
// (128^2 cavity 2.2 -> 1.16, 256^2 cavity 3.2 -> 2.1, periodic BF16 2.5 -> 1.6;
// cascaded 64^2 2.1 -> 1.12, central moments 2.0 -> 0.87, cascaded with a force
// 256^2 cavity 3.5 -> 2.9).
// Three or six steps per launch measured 0.99 and 1.03 at 64^2, eight 1.25.
// Tile sizes are compile-time constants, so that the planes' offsets are
// immediates and the divisions multiplications: with sizes as arguments 64^2
// took 1.09 and the 256^2 cavity 2.6.
template <typename S, int BC, bool FORCE, int SM, int TX, int TY, int T, int NTH>
__global__ void __launch_bounds__(NTH) k_tile(LbParams P, const S* __restrict__ fin,
                                                       const S* __restrict__ gin,
                                                       S* __restrict__ fout, S* __restrict__ gout,
                                                       const DevStatus* __restrict__ status) {
  constexpr int EX[9] = {0, 1, 0, -1, 0, 1, -1, -1, 1};
  constexpr int EY[9] = {0, 0, 1, 0, -1, 1, 1, -1, -1};
  constexpr int OPP[9] = {0, 3, 4, 1, 2, 7, 8, 5, 6};
  extern __shared__ __align__(16) unsigned char tile_shared[];
  S* const buf = reinterpret_cast<S*>(tile_shared);
  // (programmatic dependent launch: the next launch may start once every CTA is
  // here, and waits here itself; hence L2-coherent loads below)
  cudaGridDependencySynchronize();
  cudaTriggerProgrammaticLaunchCompletion();
  if (status->stopped) return;
  const int nx = P.nx, ny = P.ny;
  const int x0 = blockIdx.x * TX, y0 = blockIdx.y * TY;
  const int x1 = min(x0 + TX, nx), y1 = min(y0 + TY, ny);
  constexpr int h = T - 1, stride = TX + 2 * h;  // of the buffers' rows
  constexpr int plane = stride * (TY + 2 * h);
#pragma unroll
  for (int l = 1; l <= T; ++l) {
    const int e = T - l;
    // (the whole region's width, so that the divisions are by constants)
    const int w = TX + 2 * e, n = w * (TY + 2 * e);
    const S* const src = buf + (l & 1) * 18 * plane;
    S* const dst = buf + ((l & 1) ^ 1) * 18 * plane;
    for (int idx = threadIdx.x; idx < n; idx += NTH) {
      const int r = idx / w;
      const int X = x0 - e + idx - r * w, Y = y0 - e + r;  // (outside the lattice where it wraps)
      if (X >= x1 + e || Y >= y1 + e) continue;
      if (BC == BC_CAVITY && (X < 0 || X >= nx)) continue;
      if (BC != BC_PERIODIC && (Y < 0 || Y >= ny)) continue;
      int x = X, y = Y;
      if (BC != BC_CAVITY) x = x < 0 ? x + nx : x >= nx ? x - nx : x;
      if (BC == BC_PERIODIC) y = y < 0 ? y + ny : y >= ny ? y - ny : y;
      const int o = (Y - y0 + h) * stride + (X - x0 + h);
      float df[9], dg[9];
      if (l == 1) {
        pull<S, BC, true>(P, fin, gin, x, y, df, dg);
      } else {
        const bool sxm = BC == BC_CAVITY && x == 0, sxp = BC == BC_CAVITY && x == nx - 1;
        const bool sym = BC != BC_PERIODIC && y == 0, syp = BC != BC_PERIODIC && y == ny - 1;
        if (BC == BC_PERIODIC || !(sxm || sxp || sym || syp)) {
#pragma unroll
          for (int a = 0; a < 9; ++a) {
            const S* q = src + a * plane + o - EY[a] * stride - EX[a];
            df[a] = Codec<S>::get(q, P.isf);
            dg[a] = Codec<S>::get(q + 9 * plane, P.isg);
          }
        } else {  // the wall rules of pull()
          const bool solid[9] = {false,      sxm,        sym,        sxp,       syp,
                                 sxm || sym, sxp || sym, sxp || syp, sxm || syp};
          const bool lidl[9] = {false, false, false, false, syp, false, false, syp, syp};
#pragma unroll
          for (int a = 0; a < 9; ++a) {
            const bool bb = solid[a];
            const S* q = src + (bb ? OPP[a] * plane + o : a * plane + o - EY[a] * stride - EX[a]);
            float vf = Codec<S>::get(q, P.isf), vg = Codec<S>::get(q + 9 * plane, P.isg);
            if (bb) {
              const bool lid = lidl[a];
              vf += lid ? P.lid[a] : 0.0f;
              vg = (lid ? P.abb_lid[a] : P.abb_wall[a]) - vg;
            }
            df[a] = vf;
            dg[a] = vg;
          }
        }
      }
      collide<FORCE, SM, sizeof(S) == 4>(P, x, y, df, dg);
      if (l < T) {
#pragma unroll
        for (int a = 0; a < 9; ++a) {
          Codec<S>::put(dst + a * plane + o, df[a], P.sf);
          Codec<S>::put(dst + (a + 9) * plane + o, dg[a], P.sg);
        }
      } else {
        const uint32_t out = (uint32_t)y * (uint32_t)P.pitch + (uint32_t)x;
#pragma unroll
        for (int a = 0; a < 9; ++a) {
          Codec<S>::put(fout + a * P.plane + out, df[a], P.sf);
          Codec<S>::put(gout + a * P.plane + out, dg[a], P.sg);
        }
      }
    }
    __syncthreads();
  }
}

namespace tile {

template <typename S, int BC, bool FORCE, int SM, int TX, int TY, int NTH>
cudaError_t go(const Launch& L, const void* fin, const void* gin, void* fout, void* gout,
               const DevStatus* st) {
  constexpr int T = kTileSteps;
  auto* kernel = k_tile<S, BC, FORCE, SM, TX, TY, T, NTH>;
  // two buffers of the tile with T - 1 nodes around it
  const int smem = 2 * 18 * (TX + 2 * T - 2) * (TY + 2 * T - 2) * (int)sizeof(S);
  static SharedLimit limit;
  const cudaError_t e = limit.raise((const void*)kernel, smem);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((L.P.nx + TX - 1) / TX, (L.P.ny + TY - 1) / TY);
  cfg.blockDim = dim3(NTH);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = L.stream;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, L.P, (const S*)fin, (const S*)gin, (S*)fout, (S*)gout,
                            st);
}

template <typename S, int BC, bool FORCE, int SM>
cudaError_t go_shape(const Launch& L, const void* fin, const void* gin, void* fout, void* gout,
                     const DevStatus* st, int shape) {
  switch (shape) {
    case 0: return go<S, BC, FORCE, SM, 8, 4, 160>(L, fin, gin, fout, gout, st);
    case 1: return go<S, BC, FORCE, SM, 8, 8, 256>(L, fin, gin, fout, gout, st);
    case 2: return go<S, BC, FORCE, SM, 16, 8, 320>(L, fin, gin, fout, gout, st);
    case 3: return go<S, BC, FORCE, SM, 16, 16, 512>(L, fin, gin, fout, gout, st);
    default: return go<S, BC, FORCE, SM, 32, 14, 768>(L, fin, gin, fout, gout, st);
  }
}

template <typename S, int BC, int SM>
cudaError_t go_force(const Launch& L, const void* fin, const void* gin, void* fout, void* gout,
                     const DevStatus* st, int shape) {
  return L.force ? go_shape<S, BC, true, SM>(L, fin, gin, fout, gout, st, shape)
                 : go_shape<S, BC, false, SM>(L, fin, gin, fout, gout, st, shape);
}

template <typename S, int SM>
cudaError_t go_bc(const Launch& L, const void* fin, const void* gin, void* fout, void* gout,
                  const DevStatus* st, int shape) {
  switch (L.P_bc) {
    case BC_PERIODIC: return go_force<S, BC_PERIODIC, SM>(L, fin, gin, fout, gout, st, shape);
    case BC_CAVITY: return go_force<S, BC_CAVITY, SM>(L, fin, gin, fout, gout, st, shape);
    default: return go_force<S, BC_CHANNEL, SM>(L, fin, gin, fout, gout, st, shape);
  }
}

}  // namespace tile
}  // namespace ddflb
