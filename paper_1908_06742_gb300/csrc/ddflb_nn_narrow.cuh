// 3x3 convolutions with few input channels (16, 32 or 64) on the 5th-generation
// tensor cores, straight from the NHWC activation (included by ddflb_nn.cu).
//
// With few channels a convolution is bound by how its operand reaches shared
// memory, not by arithmetic: one TMA box per tap re-reads every pixel nine times
// and TMA takes about 3 cycles per pixel row, and an im2col matrix is nine times
// the activation.  Here a tile's pixels and their halo are copied once (16-byte
// cp.async, zeros outside the image) into planes of 8 channels, [plane][pixel] x
// 16 bytes: the core-matrix order of the K-major layout without swizzle (8 rows
// x 16 bytes contiguous, groups of 8 rows 128 bytes apart, the two K groups one
// plane apart).  Pixel rows are contiguous, so the operand of any tap is the same
// tile read from another start address, and the whole K loop (9 taps, 16 channels
// per instruction) runs from one copy.  The weights stay in shared memory.
//
// A unit is 128 consecutive positions, the rows of one MMA: a row segment where
// the width is a multiple of 128, else positions of the image with rows padded to
// width + 2, whose two extra columns are computed and dropped.  A tile is one
// unit, or two (the segments of two rows, copied with their halo as 4 x 130
// pixels instead of twice 3 x 130) where there are enough of them: the copies are
// what bounds the kernel.
//
// Measured, B = 16, BF16 out, us: 256^2 32 -> 32 61 (im2col + GEMM 330), 64 -> 32
// 97 (per-tap TMA boxes 201), 128^2 64 -> 64 37.6 (57.5).  On the way, 256^2
// 32 -> 32: four copying warps with a serial index chain 131, independent
// iterations 84, bias from shared memory and paired conversions in the epilogue
// 89 (64 -> 64: 61 -> 45), arrivals by the copies themselves 75, two units per
// tile 61.  Without the copies it takes 46, near the 65 cycles that an MMA of
// M = 128 takes whatever N is.
//
// Roles: warps 0-7 copy, warp 8 issues the MMAs, two groups of four warps store every other unit.  Every wait is
// bounded, as in the GEMM kernels.  Order of summation: taps, then channels, 16
// at a time, as im2col + GEMM (bit-identical).
//
// SEP: the adjoint for the input gradient, dX[p] = sum over taps of (g[p - tap] .
// W[tap]), with every tap's product rounded on its own and the nine summed in
// order, as the GEMM + col2im pair does it (bit-identical) without its FP32
// matrix of 9 C columns: the taps' accumulators go round a ring of 16 slots of 32
// columns in tensor memory and the epilogue adds them up in registers.
#pragma once

namespace narrow {

constexpr int CW = 8;  // copying warps
constexpr int THREADS = 32 * (CW + 9);
constexpr int SLOTS = 16;  // SEP: accumulator slots

struct Args {
  const bf16* X;  // NHWC, channel stride cs
  int B, H, W, cs;
  const bf16* Wt;     // forward: [N][9][C]; SEP: [C][9][N]
  uint32_t inv_pitch; // ceil(2^32 / pitch)
  int pitch, npos;    // positions per tile row, positions copied per tile
  int segment;        // W is a multiple of 128
  int tiles, per_img; // tiles in all (per N tile) and per image
  int unit_step;      // positions from a tile's first unit to its second
  int ntn;            // N tiles
  int nbuf;
  GemmArgs g;  // epilogue: Cf, Cb, ldc, ldcb, bias, act, accumulate, N
};

// K-major operand without swizzle: lbo between the two K groups, sbo between 8-row groups
__device__ __forceinline__ uint64_t desc_plain(uint32_t addr, uint32_t lbo, uint32_t sbo) {
  return (uint64_t)((addr & 0x3FFFFu) >> 4) | ((uint64_t)((lbo >> 4) & 0x3FFFu) << 16) |
         ((uint64_t)((sbo >> 4) & 0x3FFFu) << 32) | ((uint64_t)1 << 46);
}

template <int CH, int BN, bool SEP, int MT>  // CH: planes of 8 channels; MT: units per tile
__global__ void __launch_bounds__(THREADS, 1) k_conv_narrow(const Args a) {
  constexpr uint32_t COLS = SEP ? 512 : 2 * MT * BN;
  constexpr int NACC = SEP ? SLOTS : 2 * MT;  // accumulators
  constexpr int AW = SEP ? 32 : BN;      // columns of one
  constexpr uint32_t IDESC = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(BN >> 3) << 17) |
                             (8u << 24);
  extern __shared__ __align__(1024) uint8_t nsmem[];
  __shared__ __align__(8) uint64_t s_bars[2 * 4 + 2 * NACC + 1];
  __shared__ uint32_t s_tmem;
  __shared__ int s_abort;
  __shared__ float s_bias[BN];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const uint32_t plane = (uint32_t)a.npos * 16, bufb = CH * plane;
  const uint32_t w_u = smem_u32(nsmem), buf_u = w_u + 9 * CH * BN * 16;
  const uint32_t full_u = smem_u32(s_bars), empty_u = full_u + 32;
  const uint32_t tfull_u = full_u + 64, tempty_u = tfull_u + 8 * NACC, mdone_u = tempty_u + 8 * NACC;
  const volatile int* abort = &s_abort;
  const int n0 = (blockIdx.x % a.ntn) * BN;  // this CTA's N tile
  const int first = blockIdx.x / a.ntn, step = gridDim.x / a.ntn;

  if (tid == 0) {
    s_abort = 0;
    auto init = [](uint32_t bar, uint32_t count) {
      asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
    };
    for (int i = 0; i < a.nbuf; ++i) {
      init(full_u + 8 * i, 32 * CW);
      init(empty_u + 8 * i, 1);
    }
    for (int i = 0; i < NACC; ++i) {
      init(tfull_u + 8 * i, 1);
      init(tempty_u + 8 * i, 128);
    }
    init(mdone_u, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == CW) {
    __syncwarp();
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(&s_tmem)),
                 "r"(COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  if (tid < BN) s_bias[tid] = a.g.bias && n0 + tid < a.g.N ? a.g.bias[n0 + tid] : 0.0f;
  // the weights of all taps: [tap * CH + plane][n] x 16 bytes, zeros beyond N
  for (int i = tid; i < 9 * CH * BN; i += THREADS) {
    const int n = i % BN, kp = i / BN;  // kp = tap * CH + plane
    uint4 v = make_uint4(0u, 0u, 0u, 0u);
    if (n0 + n < a.g.N) {
      if (!SEP) {
        v = *reinterpret_cast<const uint4*>(a.Wt + ((size_t)(n0 + n) * 9 * CH + kp) * 8);
      } else {
        const int tap = kp / CH, c0 = (kp - tap * CH) * 8;
        __align__(16) bf16 h[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) h[e] = a.Wt[((size_t)(c0 + e) * 9 + tap) * a.g.N + n0 + n];
        v = *reinterpret_cast<const uint4*>(h);
      }
    }
    *reinterpret_cast<uint4*>(nsmem + (size_t)i * 16) = v;
  }
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = s_tmem;

  if (warp < CW) {
    // ---------------- copies: as many tiles in flight as there are buffers; a
    // thread's arrival on `full` fires when its copies have landed
    int issued = 0;
    for (int t = first; t < a.tiles; t += step) {
      const int b = t / a.per_img, i = t - b * a.per_img;
      const int st = issued % a.nbuf;
      if (issued >= a.nbuf && !mbar_wait_ab(empty_u + 8 * st, ((issued / a.nbuf) - 1) & 1, abort)) {
        s_abort = 1;
        break;
      }
      const uint32_t dst = buf_u + st * bufb;
      const bf16* const img = a.X + (size_t)b * a.H * a.W * a.cs;
      // This thread's plane and pixels: the lanes of a pixel read its channels
      // together.  Position q of the tile's pitch is row q / pitch.  The
      // iterations are independent, so that several are in flight: one warp a
      // scheduler does this, and a serial form of the loop was the whole
      // kernel's bound (C = 64: 200 cycles an iteration).
      constexpr int STEP = 32 * CW / CH;
      const int c = tid % CH, p0 = tid / CH;
      int q0 = p0, h0 = -1, w0 = -1;
      if (a.segment) {
        const int seg = a.W >> 7, hh = i / seg;
        h0 += hh * MT;
        w0 += (i - hh * seg) << 7;
      } else {  // (one padded row down, to stay positive)
        q0 += i * (128 * MT) - 1 + a.pitch;
        h0 -= 1;
      }
      const bf16* const srcc = img + c * 8;
      const uint32_t dstc = dst + c * plane;
#pragma unroll 8
      for (int p = p0; p < a.npos; p += STEP) {
        const uint32_t q = (uint32_t)(q0 + p - p0), r = __umulhi(q, a.inv_pitch);
        const int h = h0 + (int)r, w = w0 + (int)(q - r * a.pitch);
        const bool in = (unsigned)h < (unsigned)a.H && (unsigned)w < (unsigned)a.W;
        const bf16* src = srcc + (in ? (size_t)((h * a.W + w) * (int64_t)a.cs) : 0);
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(dstc + p * 16),
                     "l"(src), "r"(in ? 16 : 0)  // 0: zero fill
                     : "memory");
      }
      asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(full_u + 8 * st)
                   : "memory");
      ++issued;
    }
    asm volatile("cp.async.wait_all;" ::: "memory");  // nothing in flight when the CTA ends
  } else if (warp == CW) {
    // ---------------- MMA issuer: the whole warp runs the loop, so that the
    // descriptors stay in uniform registers, and one elected lane issues.  The
    // operands of a tile are one descriptor each plus offsets in 16-byte units.
    uint32_t leader;
    asm volatile(
        "{\n .reg .pred p;\n elect.sync _|p, 0xffffffff;\n selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(leader));
    int it = 0, sl = 0;  // tiles, accumulator uses (SEP: one per tap)
    bool ok = true;
    auto wait = [&](uint32_t bar, uint32_t parity) {
      return __all_sync(0xffffffffu, mbar_wait_ab(bar, parity, abort)) != 0;
    };
    auto acc_free = [&](int use) {
      return use < NACC || wait(tempty_u + 8 * (use % NACC), ((use / NACC) - 1) & 1);
    };
    auto commit = [&](uint32_t bar) {
      asm volatile(
          "{\n .reg .pred q;\n setp.ne.b32 q, %1, 0;\n"
          " @q tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n}\n" ::"r"(
              bar),
          "r"(leader)
          : "memory");
    };
    const uint64_t bd0 = desc_plain(w_u, BN * 16, 128);
    for (int t = first; t < a.tiles; t += step, ++it) {
      const int st = it % a.nbuf;
      if (!SEP) ok = acc_free(it * MT + MT - 1) && acc_free(it * MT);
      ok = ok && wait(full_u + 8 * st, (it / a.nbuf) & 1);
      if (!ok) break;
      // the copies' writes (generic proxy) before the MMAs' reads (async proxy)
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      tc_fence_after();
      const uint64_t ad0 = desc_plain(buf_u + st * bufb, plane, 128);
      // SEP: unit by unit, each tap into a slot of its own; else both units tap by tap
#pragma unroll
      for (int k = 0; k < (SEP ? 9 * MT : 9); ++k) {
        const int tap = SEP ? k % 9 : k;
        const int ty = SEP ? 2 - tap / 3 : tap / 3, tx = SEP ? 2 - tap % 3 : tap % 3;
        if (SEP) {
          ok = ok && acc_free(sl);
          if (!ok) break;
          tc_fence_after();
        }
#pragma unroll
        for (int u = 0; u < (SEP ? 1 : MT); ++u) {
          const int unit = SEP ? k / 9 : u;
          const uint32_t d = tmem + (uint32_t)(SEP ? (sl % NACC) * AW : ((it * MT + u) % NACC) * BN);
#pragma unroll
          for (int kk = 0; kk < CH / 2; ++kk) {
            const uint64_t ad =
                ad0 + (uint32_t)(unit * a.unit_step + ty * a.pitch + tx + 2 * kk * a.npos);
            const uint64_t bd = bd0 + (uint32_t)((tap * CH + 2 * kk) * BN);
            asm volatile(
                "{\n .reg .pred p, q;\n setp.ne.b32 p, %4, 0;\n setp.ne.b32 q, %5, 0;\n"
                " @q tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(d),
                "l"(ad), "l"(bd), "r"(IDESC), "r"((SEP ? kk > 0 : (tap > 0 || kk > 0)) ? 1u : 0u),
                "r"(leader)
                : "memory");
          }
        }
        if (SEP) {
          commit(tfull_u + 8 * (sl % NACC));
          ++sl;
        }
      }
      if (!ok) break;
      commit(empty_u + 8 * st);
      if (!SEP)
        for (int u = 0; u < MT; ++u) commit(tfull_u + 8 * ((it * MT + u) % NACC));
    }
    if (!ok) s_abort = 1;
    // every MMA issued has completed before the CTA moves on
    commit(mdone_u);
    if (!mbar_wait(mdone_u, 0)) s_abort = 1;
  } else {
    // ---------------- epilogue: two groups of four warps take every other unit;
    // a warp reads lane quarter q
    const int q = warp & 3, row = q * 32 + lane, group = (warp - CW - 1) >> 2;
    const bool vf = a.g.Cf && (a.g.ldc & 3) == 0 && ((uintptr_t)a.g.Cf & 15) == 0;
    const bool vb = a.g.Cb && (a.g.ldcb & 7) == 0 && ((uintptr_t)a.g.Cb & 15) == 0;
    auto ready = [&](int use) {
      int ok = 1;
      if (lane == 0) ok = mbar_wait_ab(tfull_u + 8 * (use % NACC), (use / NACC) & 1, abort) ? 1 : 0;
      return __shfl_sync(0xffffffffu, ok, 0) != 0;
    };
    auto release = [&](int use) {
      tc_fence_before();
      asm volatile("mbarrier.arrive.release.cta.shared::cta.b64 _, [%0];" ::"r"(
                       tempty_u + 8 * (use % NACC))
                   : "memory");
    };
    // unit it = tile number * MT + place in the tile
    for (int it = group;; it += 2) {
      const int t = first + (it / MT) * step, sub = it % MT;
      if (t >= a.tiles) break;
      const int b = t / a.per_img, i = t - b * a.per_img;
      int px = -1;  // output pixel of this row of the unit
      if (a.segment) {
        const int seg = a.W >> 7, hh = i / seg, h = hh * MT + sub;
        if (h < a.H) px = (b * a.H + h) * a.W + ((i - hh * seg) << 7) + row;
      } else {
        const int p = (i * MT + sub) * 128 + row, h = p / a.pitch, w = p - h * a.pitch - 1;
        if (h < a.H && w >= 0 && w < a.W) px = (b * a.H + h) * a.W + w;
      }
      const uint32_t lane_base = tmem + ((uint32_t)(q * 32) << 16);
      if (SEP) {
        float s[32];
#pragma unroll
        for (int k = 0; k < 32; ++k) s[k] = 0.0f;
        bool ok = true;
        int sl = it * 9;
#pragma unroll 1
        for (int tap = 0; tap < 9; ++tap, ++sl) {
          if (!ready(sl)) {
            ok = false;
            break;
          }
          tc_fence_after();
          uint32_t v[32];
          tmem_ld32(lane_base + (uint32_t)((sl % NACC) * AW), v);
          release(sl);
#pragma unroll
          for (int k = 0; k < 32; ++k) s[k] += __uint_as_float(v[k]);
        }
        if (!ok) {
          s_abort = 1;
          break;
        }
        uint32_t v[32];
#pragma unroll
        for (int k = 0; k < 32; ++k) v[k] = __float_as_uint(s[k]);
        if (px >= 0) store_row32(a.g, px, n0, 0, v, true, vf, vb);
      } else {
        if (!ready(it)) {
          s_abort = 1;
          break;
        }
        tc_fence_after();
#pragma unroll 1
        for (int c0 = 0; c0 < BN; c0 += 32) {
          uint32_t v[32];
          tmem_ld32(lane_base + (uint32_t)((it % NACC) * BN + c0), v);
          if (px < 0 || n0 + c0 >= a.g.N) continue;
          if (a.g.Cf || !vb || n0 + c0 + 32 > a.g.N) {
            store_row32(a.g, px, n0 + c0, 0, v, true, vf, vb);
            continue;
          }
          // BF16 output, whole chunk: bias from shared memory, paired conversions
          // (the same bits as store_row32, in a third of its instructions)
          uint4* const o = reinterpret_cast<uint4*>(a.g.Cb + (size_t)px * a.g.ldcb + n0 + c0);
#pragma unroll
          for (int k = 0; k < 32; k += 8) {
            uint32_t w[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              float x = __uint_as_float(v[k + 2 * e]), y = __uint_as_float(v[k + 2 * e + 1]);
              if (a.g.bias) {
                x += s_bias[c0 + k + 2 * e];
                y += s_bias[c0 + k + 2 * e + 1];
              }
              const __nv_bfloat162 h = __floats2bfloat162_rn(act_fwd(x, a.g.act), act_fwd(y, a.g.act));
              w[e] = *reinterpret_cast<const uint32_t*>(&h);
            }
            o[k / 8] = make_uint4(w[0], w[1], w[2], w[3]);
          }
        }
        release(it);
      }
    }
  }
  __syncwarp();
  __syncthreads();
  if (s_abort && tid == 0) atomicExch(&g_tc_error, 1);
  tc_fence_before();
  __syncthreads();
  if (warp == CW) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(COLS)
                 : "memory");
  }
}

}  // namespace narrow
