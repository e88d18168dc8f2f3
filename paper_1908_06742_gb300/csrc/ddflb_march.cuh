// Two fused time steps per pass over memory (k_march2), one warp per strip of
// the lattice: see the kernel's comment.  Included by one translation unit per
// storage type and model, so that they compile in parallel.
#pragma once

#include <cuda_runtime.h>

#include "ddflb_device.cuh"
#include "ddflb_internal.h"
#include "ddflb_pair.cuh"

namespace ddflb {

// A lane owns two adjacent columns (the first one even): FP32 pairs are 8-byte
// words, 16-bit pairs 4-byte words.
template <typename S> struct PairIo;

template <> struct PairIo<float> {
  static constexpr int ALIGN = 4, SEG = 68, STAGES = 2;  // elements per 16 bytes, per staged row
  static __device__ __forceinline__ F2 ld(const float* p) {
    return *reinterpret_cast<const float2*>(p);
  }
  static __device__ __forceinline__ F2 ld1(const float* p) { return make_float2(p[0], p[1]); }
  static __device__ __forceinline__ void st_global(float* p, F2 v) {
    __stcs(reinterpret_cast<float2*>(p), v);
  }
  static __device__ __forceinline__ void st(float* p, F2 v) { *reinterpret_cast<float2*>(p) = v; }
  static __device__ __forceinline__ F2 round(F2 v) { return v; }
};

template <typename S> struct PairIo {
  static constexpr int ALIGN = 8, SEG = 72, STAGES = 3;
  static __device__ __forceinline__ F2 ld(const S* p) {
    return widen<S>(*reinterpret_cast<const unsigned*>(p));
  }
  static __device__ __forceinline__ F2 ld1(const S* p) {
    return make_float2(widen1(p[0]), widen1(p[1]));
  }
  static __device__ __forceinline__ void st_global(S* p, F2 v) {
    __stcs(reinterpret_cast<unsigned*>(p), narrow<S>(v));
  }
  static __device__ __forceinline__ void st(S* p, F2 v) {
    *reinterpret_cast<unsigned*>(p) = narrow<S>(v);
  }
  // populations between the two steps are rounded to the storage type, as if stored
  static __device__ __forceinline__ F2 round(F2 v) { return widen<S>(narrow<S>(v)); }
};

__device__ __forceinline__ uint32_t shared_addr(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}

// Bounded wait for an mbarrier phase: about a second at most.
__device__ __forceinline__ bool phase_wait(uint32_t bar, uint32_t parity) {
  for (uint32_t it = 0; it < (1u << 20); ++it) {
    uint32_t done;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, 1000;\n"
        " selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(done)
        : "r"(bar), "r"(parity)
        : "memory");
    if (done) return true;
  }
  return false;
}

__device__ __forceinline__ int dir_ey(int a) {
  return a == 2 || a == 5 || a == 6 ? 1 : a == 4 || a == 7 || a == 8 ? -1 : 0;
}

// The pair of values that the two columns pull from x - 1 (from_left) or x + 1.
__device__ __forceinline__ F2 from_left(F2 v) {
  return make_float2(__shfl_up_sync(0xffffffffu, v.y, 1), v.x);
}
__device__ __forceinline__ F2 from_right(F2 v) {
  return make_float2(v.y, __shfl_down_sync(0xffffffffu, v.x, 1));
}

// warps per SM (the register budget: 128 at 16, 168 at 12)
template <typename S, int BC, bool FORCE = false, int SM = 0>
constexpr int kMarchWarps = (sizeof(S) == 4 && BC != BC_PERIODIC) || FORCE || SM ? 12 : 16;

template <typename S>
constexpr size_t march_smem(int bc) {
  // the staged rows, three rows of values handed on (6 planes each) and, with
  // walls, the e_y = -1 values of one row
  return (size_t)(PairIo<S>::STAGES * 18 * PairIo<S>::SEG + 18 * 64) * sizeof(S) +
         (bc != BC_PERIODIC ? 6 * 64 * sizeof(S) : 0);
}

// One warp marches up a strip of 64 columns (60 of them its own, two on each
// side computed for its neighbours' sake), a chunk of `rows` rows.  In
// iteration i it takes row i through the first step and row i - 1 through the
// second, so the lattice crosses memory once per two steps (72 B per node and
// step at FP32 instead of 144).
//
// Why this shape: with half the traffic the step is bound by FP32 issue, so
// what counts is instructions per node and warps that never wait for each
// other.  The arithmetic is packed (ddflb_pair.cuh); the source rows arrive by
// bulk copies one or two rows ahead, which costs no address arithmetic and hides
// DRAM; the values a row hands to the rows above live in the warp's own shared
// memory, so there is no block barrier.  Forms measured on the way, FP32 8192^2,
// thousand million node updates a second (k_step: 46.0): CTAs of 128 threads
// over a shared ring, scalar arithmetic 57, packed 59, packed and fed by bulk
// copies 65; one warp per strip with the rows handed on in registers (163, so
// 3 warps per scheduler) 76; in shared memory (126 registers, 4 per scheduler)
// 79, 311 instructions per node and step against 553.  FP16 16384^2: 108 against
// 91 of k_step_quad (16 warps an SM; 12: 97, 20 with spills: 78).  The walled
// FP32 forms keep 12 warps (4096^2 cavity: 67; at 16, with spills: 60), and so do
// those with a force or a central-moment model (8192 x 4096 periodic, us per step,
// two nodes per thread -> this: forced MRT 691 -> 501, cascaded 695 -> 557, forced
// cascaded 703 -> 605, central moments 691 -> 524).
//
// `strip` and rows [y0, y1) name the strip and chunk; shared: march_smem() bytes;
// bars: STAGES mbarriers; wall: 12 floats.  If a copy does not arrive, the rest of the
// chunk is not written and *stop, 0 until then, takes `bit` (a plain store: the same
// from every warp; an atomic cost the cavity forms registers).
template <typename S, int BC, bool FORCE = false, int SM = 0>
__device__ __forceinline__ void march_strip(const LbParams& P, const PairConst& K,
                                            const S* __restrict__ fin, const S* __restrict__ gin,
                                            S* __restrict__ fout, S* __restrict__ gout, int strip,
                                            int y0, int y1, unsigned char* shared, uint64_t* bars,
                                            float* s_wall, int* stop, int bit) {
  using Io = PairIo<S>;
  constexpr bool COMP = sizeof(S) == 4;
  static_assert(COMP || !(FORCE || SM), "16-bit storage: unforced MRT only");
  // the force is the same at every node and step
  const F2 Fx = make_float2(P.fx * P.fmod, P.fx * P.fmod);
  const F2 Fy = make_float2(P.fy * P.fmod, P.fy * P.fmod);
  constexpr int NST = Io::STAGES, SEG = Io::SEG, W = kMarchStrip;
  S* const stage0 = reinterpret_cast<S*>(shared);
  // stage 0, the values handed on, the other stages, D: the outer lanes' reads one
  // element beside the handed-on planes stay inside (and without margins 15
  // periodic FP32 warps fit an SM)
  auto stage_at = [&](int k) { return stage0 + k * 18 * SEG + (k > 0 ? 18 * 64 : 0); };
  // values handed on: [6][64] e_y = 0 of row i - 1 (lattice * 3 + k: directions 0,
  // 1, 3), [2][6][64] e_y = +1 (2, 5, 6) of rows i - 1 and i - 2 by the row's
  // parity; with walls [6][64] e_y = -1 (4, 7, 8) of row i - 1
  S* const E = stage0 + 18 * SEG + 2 * threadIdx.x;
  S* const U = E + 6 * 64;
  S* const D = stage0 + NST * 18 * SEG + 18 * 64 + 2 * threadIdx.x;
  const int lane = threadIdx.x;
  const int nx = P.nx, ny = P.ny;
  // the strip's 64 columns from xl; its own are [xs, xe).  A cavity has no columns
  // beyond its walls, so there the first strip starts at the wall and the last
  // one ends at it.
  const int xl = BC == BC_CAVITY ? strip * W : strip * W - 2;
  const int xs = BC == BC_CAVITY && strip == 0 ? 0 : xl + 2;
  const bool left = strip == 0;
  const bool right = BC == BC_CAVITY ? xl + 64 >= nx : xl + 64 > nx;
  const int xe = BC == BC_CAVITY ? (right ? nx : xl + 62) : min(xs + W, nx);
  const bool inside = !left && !right;  // nothing of it is at an edge of the lattice
  const int xa = xl + 2 * lane;         // this lane's columns: xa, xa + 1
  // the staged segment (from a 16-byte boundary), cut to the row
  const int seg0 = (xl - 1) & ~(Io::ALIGN - 1);  // (may be negative)
  const int segb = max(seg0, 0), sege = min(seg0 + SEG, P.pitch);
  const uint32_t seg = (uint32_t)(sege - segb) * (uint32_t)sizeof(S);
  const uint32_t bar0 = shared_addr(bars);
  if (lane < NST)
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar0 + 8 * lane) : "memory");
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  __syncwarp();

  // row i is pulled from the stage (else, next to a wall, straight from memory)
  auto staged = [&](int i) { return i <= y1 && (BC == BC_PERIODIC || (i >= 1 && i < ny - 1)); };
  // lane a (18 lanes) copies its plane's segment of row i - e_y
  const int pa = lane < 9 ? lane : lane - 9;
  const S* const psrc = (lane < 9 ? fin : gin) + (lane < 18 ? pa : 0) * P.plane + segb;
  const int pey = dir_ey(pa);
  const uint32_t pdst = shared_addr(stage0 + (lane < 18 ? lane : 0) * SEG + (segb - seg0));
  auto fetch = [&](int i, int st) {
    const uint32_t bar = bar0 + 8 * st;
    if (lane == 0)
      asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar),
                   "r"(18 * seg)
                   : "memory");
    __syncwarp();
    if (lane < 18) {
      int y = i - pey;
      if (BC == BC_PERIODIC) {
        if (y < 0) y += ny;
        else if (y >= ny) y -= ny;
      }
      asm volatile(
          "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, "
          "[%3];" ::"r"(pdst + (uint32_t)((st * 18 * SEG + (st > 0 ? 18 * 64 : 0)) * (int)sizeof(S))),
          "l"(psrc + (int64_t)y * P.pitch), "r"(seg), "r"(bar)
          : "memory");
    }
  };
  // What the staged rows lack at the lattice's sides, loaded one row ahead into
  // registers: the two columns beyond a periodic side (copies of those they wrap
  // to: 18 planes x 2 columns a side), or the own values of the opposite
  // directions that a side wall bounces back (3 directions x 2 lattices a side).
  constexpr int NEDGE = BC == BC_CAVITY ? 1 : 3;
  S edge[NEDGE];
  auto fetch_edge = [&](int i) {
    if (BC == BC_CAVITY) {
      const int side = lane / 6, k = lane % 6;  // k: lattice * 3 + direction
      if (lane < 12 && (side ? right : left)) {
        const int a = side ? (k % 3 == 0 ? 1 : k % 3 == 1 ? 8 : 5)   // opposites of 3, 6, 7
                           : (k % 3 == 0 ? 3 : k % 3 == 1 ? 7 : 6);  // opposites of 1, 5, 8
        edge[0] = __ldg((k < 3 ? fin : gin) + a * P.plane + (int64_t)i * P.pitch +
                        (side ? nx - 1 : 0));
      }
    } else {
#pragma unroll
      for (int j = 0; j < NEDGE; ++j) {
        const int e = lane + 32 * j, side = e / 36, p = e % 36 >> 1, c = e & 1;
        if (e < 72 && (side ? right : left)) {
          const int a = p < 9 ? p : p - 9;
          int y = i - dir_ey(a);
          if (BC == BC_PERIODIC) {
            if (y < 0) y += ny;
            else if (y >= ny) y -= ny;
          }
          const int x = side ? (c < nx ? c : 0) : max(nx - 2 + c, 0);
          edge[j] = __ldg((p < 9 ? fin : gin) + a * P.plane + (int64_t)y * P.pitch + x);
        }
      }
    }
  };
  auto put_edge = [&](int st) {
    if (BC == BC_CAVITY) {
      const int side = lane / 6, k = lane % 6;
      if (lane < 12 && (side ? right : left)) {
        const int a = side ? (k % 3 == 0 ? 3 : k % 3 == 1 ? 6 : 7)
                           : (k % 3 == 0 ? 1 : k % 3 == 1 ? 5 : 8);
        const float v = k < 3 ? Codec<S>::get(edge, P.isf) + 0.0f
                              : P.abb_wall[a] - Codec<S>::get(edge, P.isg);
        s_wall[side * 6 + k] = COMP ? v : v * (k < 3 ? P.sf : P.sg);
      }
    } else {
#pragma unroll
      for (int j = 0; j < NEDGE; ++j) {
        const int e = lane + 32 * j, side = e / 36, p = e % 36 >> 1, c = e & 1;
        if (e < 72 && (side ? right : left))
          stage_at(st)[p * SEG + (side ? nx + c : c - 2) - seg0] = edge[j];
      }
      // (the next copy into this stage goes through the async proxy)
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    __syncwarp();
  };
  const int first = BC == BC_PERIODIC ? y0 - 1 : max(y0 - 1, 1);  // first staged row
  for (int k = 0; k < NST; ++k)
    if (staged(first + k)) fetch(first + k, k);
  if (!inside && staged(first)) fetch_edge(first);

  int st = 0;
  uint32_t phase = 0;
  bool bad = false;
  S* up = U;  // slot of row i (and, until it is written, of row i - 2)
  S* up1 = U + 6 * 64;  // slot of row i - 1
  for (int i = y0 - 1; i <= y1; ++i) {
    F2 df[9], dg[9];
    // ---- first step, row i
    const bool exists = BC == BC_PERIODIC || (i >= 0 && i < ny);
    if (exists) {
      const bool sg = staged(i);
      if (sg) {
        if (__any_sync(0xffffffffu, !phase_wait(bar0 + 8 * st, phase))) {
          bad = true;
          break;
        }
        if (!inside) put_edge(st);
        const S* const s = stage_at(st) + (xl - seg0) + 2 * lane;
#pragma unroll
        for (int l = 0; l < 2; ++l) {
          F2* d = l ? dg : df;
          const S* q = s + l * 9 * SEG;
          d[0] = Io::ld(q);
          d[1] = Io::ld1(q + SEG - 1);
          d[2] = Io::ld(q + 2 * SEG);
          d[3] = Io::ld1(q + 3 * SEG + 1);
          d[4] = Io::ld(q + 4 * SEG);
          d[5] = Io::ld1(q + 5 * SEG - 1);
          d[6] = Io::ld1(q + 6 * SEG + 1);
          d[7] = Io::ld1(q + 7 * SEG + 1);
          d[8] = Io::ld1(q + 8 * SEG - 1);
        }
        if (BC == BC_CAVITY && !inside) {
#pragma unroll
          for (int l = 0; l < 2; ++l) {
            F2* d = l ? dg : df;
            const float* const w = s_wall + 3 * l;
            if (xa == 0) d[1].x = w[0], d[5].x = w[1], d[8].x = w[2];
            if (xa == nx - 1) d[3].x = w[6], d[6].x = w[7], d[7].x = w[8];
            if (xa + 1 == nx - 1) d[3].y = w[6], d[6].y = w[7], d[7].y = w[8];
          }
        }
      }
      if (!sg) {
        // a row next to a wall: node by node from memory
#pragma unroll 1
        for (int k = 0; k < 2; ++k) {
          int x = xa + k;
          bool live = x >= xs - 1 && x <= xe;
          if (BC == BC_CAVITY) live = live && x >= 0 && x < nx;
          else if (x < 0) x += nx;
          else if (x >= nx) x -= nx;
          if (live) {
            float vf[9], vg[9];
            pull<S, BC>(P, fin, gin, x, i, vf, vg);
#pragma unroll
            for (int a = 0; a < 9; ++a) {  // in storage units (a power of two: exact)
              const float f = COMP ? vf[a] : vf[a] * P.sf, g = COMP ? vg[a] : vg[a] * P.sg;
              if (k) df[a].y = f, dg[a].y = g;
              else df[a].x = f, dg[a].x = g;
            }
          }
        }
      }
      collide_pair<COMP, FORCE, SM>(K, df, dg, Fx, Fy);
      if (sg) {
        // every lane has read this stage: refill it
        __syncwarp();
        if (staged(i + NST)) fetch(i + NST, st);
        if (!inside && staged(i + 1)) fetch_edge(i + 1);
        if (++st == NST) {
          st = 0;
          phase ^= 1;
        }
      }
#pragma unroll
      for (int a = 0; a < 9; ++a) {
        if (dir_ey(a) >= 0) continue;
        df[a] = Io::round(df[a]);
        dg[a] = Io::round(dg[a]);
      }
    }
    // ---- second step, row i - 1
    const int y = i - 1;
    F2 nf[9], ng[9];
#pragma unroll
    for (int l = 0; l < 2; ++l) {
      F2* n = l ? ng : nf;
      const F2* d = l ? dg : df;
      const S *e = E + l * 3 * 64, *u = up + l * 3 * 64;
      n[0] = Io::ld(e);
      n[1] = Io::ld1(e + 64 - 1);
      n[3] = Io::ld1(e + 2 * 64 + 1);
      n[2] = Io::ld(u);
      n[5] = Io::ld1(u + 64 - 1);
      n[6] = Io::ld1(u + 2 * 64 + 1);
      n[4] = d[4];
      n[7] = from_right(d[7]);
      n[8] = from_left(d[8]);
    }
    if (y >= y0) {
      if (BC != BC_PERIODIC && (y == 0 || y == ny - 1 || (BC == BC_CAVITY && !inside))) {
        // the wall rules of pull(): the own value of the opposite direction,
        // with the moving-wall term, or 2 w phi_w minus it
        const bool sym = y == 0, syp = y == ny - 1;
#pragma unroll 1
        for (int k = 0; k < 2; ++k) {
          const int x = xa + k;
          const bool sxm = BC == BC_CAVITY && x == 0, sxp = BC == BC_CAVITY && x == nx - 1;
          const bool solid[9] = {false,      sxm,        sym,        sxp,       syp,
                                 sxm || sym, sxp || sym, sxp || syp, sxm || syp};
          const bool lidl[9] = {false, false, false, false, syp, false, false, syp, syp};
          // own value of direction b of lattice l in row i - 1, physical units
          auto own = [&](int l, int b) {
            const S* q = dir_ey(b) == 0 ? E + (l * 3 + (b == 1 ? 1 : 2)) * 64
                         : dir_ey(b) > 0 ? up1 + (l * 3 + (b == 2 ? 0 : b == 5 ? 1 : 2)) * 64
                                         : D + (l * 3 + (b == 4 ? 0 : b == 7 ? 1 : 2)) * 64;
            return Codec<S>::get(q + k, l ? P.isg : P.isf);
          };
          constexpr int OPP[9] = {0, 3, 4, 1, 2, 7, 8, 5, 6};
#pragma unroll
          for (int a = 1; a < 9; ++a) {
            if (solid[a]) {
              const bool lid = lidl[a];
              float vf = own(0, OPP[a]), vg = own(1, OPP[a]);
              vf += lid ? P.lid[a] : 0.0f;
              vg = (lid ? P.abb_lid[a] : P.abb_wall[a]) - vg;
              if (!COMP) vf *= P.sf, vg *= P.sg;
              if (k) nf[a].y = vf, ng[a].y = vg;
              else nf[a].x = vf, ng[a].x = vg;
            }
          }
        }
      }
    }
    __syncwarp();  // every lane has read rows i - 1 and i - 2: row i replaces them
#pragma unroll
    for (int l = 0; l < 2; ++l) {
      const F2* d = l ? dg : df;
      S *e = E + l * 3 * 64, *u = up + l * 3 * 64;
      Io::st(e, d[0]);
      Io::st(e + 64, d[1]);
      Io::st(e + 2 * 64, d[3]);
      Io::st(u, d[2]);
      Io::st(u + 64, d[5]);
      Io::st(u + 2 * 64, d[6]);
      if (BC != BC_PERIODIC) {
        S* q = D + l * 3 * 64;
        Io::st(q, d[4]);
        Io::st(q + 64, d[7]);
        Io::st(q + 2 * 64, d[8]);
      }
    }
    __syncwarp();
    if (y >= y0) {
      collide_pair<COMP, FORCE, SM>(K, nf, ng, Fx, Fy);
      if (xa >= xs && xa < xe) {
        // (where nx is odd the last pair's second value lands in the row's padding)
        const int64_t o = (int64_t)y * P.pitch + xa;
#pragma unroll
        for (int a = 0; a < 9; ++a) {
          Io::st_global(fout + a * P.plane + o, nf[a]);
          Io::st_global(gout + a * P.plane + o, ng[a]);
        }
      }
    }
    S* const t = up;
    up = up1;
    up1 = t;
  }
  if (bad) {
    // a copy did not arrive: let those in flight land (bounded), then report
    for (int k = 0; k < NST; ++k) {
      phase_wait(bar0 + 8 * st, phase);
      if (++st == NST) {
        st = 0;
        phase ^= 1;
      }
    }
    if (lane == 0) *stop = bit;
  }
}

template <typename S, int BC, bool FORCE, int SM>
__global__ void __launch_bounds__(32, kMarchWarps<S, BC, FORCE, SM>)
    k_march2(LbParams P, PairConst K, const S* __restrict__ fin, const S* __restrict__ gin,
             S* __restrict__ fout, S* __restrict__ gout, DevStatus* __restrict__ status,
             int rows) {
  extern __shared__ __align__(16) unsigned char march_shared[];
  __shared__ __align__(8) uint64_t s_bar[PairIo<S>::STAGES];
  __shared__ float s_wall[12];  // cavity: the side walls' links in row i
  if (status->stopped) return;
  const int y0 = blockIdx.y * rows;
  march_strip<S, BC, FORCE, SM>(P, K, fin, gin, fout, gout, blockIdx.x, y0, min(y0 + rows, P.ny),
                                march_shared, s_bar, s_wall, &status->stopped, kStopTimeout);
}

namespace march {

template <typename S, int BC, bool FORCE, int SM>
cudaError_t go(const Launch& L, const void* fin, const void* gin, void* fout, void* gout,
               DevStatus* st, int rows) {
  const dim3 g(march_strips(BC, L.P.nx), (L.P.ny + rows - 1) / rows);
  k_march2<S, BC, FORCE, SM><<<g, 32, march_smem<S>(BC), L.stream>>>(
      L.P, make_pair_const(L.P), (const S*)fin, (const S*)gin, (S*)fout, (S*)gout, st, rows);
  return cudaGetLastError();
}

template <typename S, bool FORCE, int SM>
cudaError_t go_bc(const Launch& L, const void* fin, const void* gin, void* fout, void* gout,
                  DevStatus* st, int rows) {
  switch (L.P_bc) {
    case BC_PERIODIC: return go<S, BC_PERIODIC, FORCE, SM>(L, fin, gin, fout, gout, st, rows);
    case BC_CAVITY: return go<S, BC_CAVITY, FORCE, SM>(L, fin, gin, fout, gout, st, rows);
    default: return go<S, BC_CHANNEL, FORCE, SM>(L, fin, gin, fout, gout, st, rows);
  }
}

}  // namespace march
}  // namespace ddflb
