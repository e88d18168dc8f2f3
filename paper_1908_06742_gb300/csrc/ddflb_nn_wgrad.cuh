// Weight gradient of a 3x3 convolution, straight from the NHWC activation and
// the NHWC output gradient (included by ddflb_nn.cu):
//   dW[co][tap][ci] = sum over pixels p of g[p][co] x[p + tap][ci].
//
// The contraction runs over pixels, so both operands are needed with the
// channels along M and N: the planes of 8 channels of the narrow convolutions
// ([plane][pixel] x 16 bytes) are also the MN-major core-matrix order without
// swizzle (8 pixels x 8 channels per core matrix, pixels 16 bytes apart), with the
// strides' roles exchanged.  There is no transposed im2col matrix and no
// transposed gradient: a unit is 64 consecutive positions (of a row where the
// width is a multiple of 64, else of the image with rows padded to width + 2 and
// zeros there), copied once with one pixel more on each side, and the three taps
// of a kernel row are three start addresses in it.
//
// A CTA takes one slice of the pixels, one kernel row and one tile of input
// channels, sums its units into three accumulators in tensor memory and writes
// them as a slice of a split-K sum, which k_splitk_reduce adds in a fixed order.
// The slices are those of the GEMM on the im2col matrix, and where the width is a
// multiple of 64 so is the order of the pixels: bit-identical to it.  (The order
// matters: a sum of thousands of pixels in one accumulator is 1e-5 off, and
// another slicing would differ by as much.)  M is always 128: the rows beyond Co
// read whatever follows the gradient in shared memory and are never stored.
//
// Bound by the MMAs (65 cycles for M = 128, K = 16 whatever N is) on the large
// levels and by the latency of few CTAs on the small ones.  B = 16, us, with the
// slice sum: 128^2 32 -> 32 55 (transposes, im2col and GEMM 128; the MMAs alone
// 31), 64 -> 32 72 (223), 64^2 64 -> 64 41 (84).  All nine taps in one CTA with
// slices of its own was faster on the small levels (370 against 566 us over the
// network) but 9e-6 off the GEMM's sums.
#pragma once

namespace wgrad {

constexpr int UNIT = 64;
constexpr int CW = 8;  // copying warps
constexpr int MAXBUF = 8;
constexpr int THREADS = 32 * (CW + 1 + 4);

struct Args {
  const bf16 *X, *G;  // NHWC, channel strides csx, csg
  int H, W, csx, csg, Ci, Co;
  uint32_t inv_pitch;
  int pitch, segment;
  int units, per_img, per_slice;  // in all, per image, per slice
  int ntn, nbuf;
  int lanes, lane_bits;  // a power of two >= Co / 8
  float* partial;  // [slice][Co][9 Ci]
};

template <int CHX>  // planes of x per N tile: 2 (Ci = 16) or 4
__global__ void __launch_bounds__(THREADS, 2) k_conv_wgrad(const Args a) {
  constexpr int BN = 8 * CHX;
  constexpr uint32_t COLS = 128;  // three accumulators
  // as the other kernels, with both operands MN-major (bits 15, 16)
  constexpr uint32_t IDESC = (1u << 4) | (1u << 7) | (1u << 10) | (1u << 15) | (1u << 16) |
                             ((uint32_t)(BN >> 3) << 17) | (8u << 24);
  extern __shared__ __align__(1024) uint8_t nsmem[];
  __shared__ __align__(8) uint64_t s_bars[2 * MAXBUF + 1];
  __shared__ uint32_t s_tmem;
  __shared__ int s_abort;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int chg = a.Co >> 3;
  constexpr uint32_t GPLANE = UNIT * 16;
  constexpr uint32_t XPLANE = (UNIT + 2) * 16;
  const uint32_t gbytes = (uint32_t)chg * GPLANE, bufb = gbytes + CHX * XPLANE;
  const uint32_t buf_u = smem_u32(nsmem);
  const uint32_t full_u = smem_u32(s_bars), empty_u = full_u + 8 * MAXBUF, done_u = full_u + 16 * MAXBUF;
  const volatile int* abort = &s_abort;
  const int dy = blockIdx.x % 3, nt = blockIdx.x / 3 % a.ntn, slice = blockIdx.x / (3 * a.ntn);
  const int u0 = slice * a.per_slice, u1 = min(u0 + a.per_slice, a.units);

  if (tid == 0) {
    s_abort = 0;
    for (int i = 0; i < a.nbuf; ++i) {
      asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(full_u + 8 * i), "r"(32 * CW)
                   : "memory");
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(empty_u + 8 * i) : "memory");
    }
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(done_u) : "memory");
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
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = s_tmem;

  if (warp < CW) {
    // ---------------- copies (see k_conv_narrow)
    // (the unit's image, place and buffer advance without divisions: with the
    // copies' own indices they are what these warps are bound by)
    int b = u0 / a.per_img, i = u0 - b * a.per_img, st = 0, round = 0;
    const int seg = a.segment ? a.W / UNIT : 1;
    int hh = i / seg, sg = i - hh * seg;
    for (int t = u0; t < u1; ++t) {
      if (round > 0 && !mbar_wait_ab(empty_u + 8 * st, (round - 1) & 1, abort)) {
        s_abort = 1;
        break;
      }
      const uint32_t dst = buf_u + st * bufb;
      const size_t img = (size_t)b * a.H * a.W;
      // positions of the unit's row or of the padded image: the gradient's start at
      // qg, the activation's (one kernel row of taps) at qx
      int qg = 0, qx = -1, h0 = 0, w0 = 0;
      if (a.segment) {
        h0 = hh;
        w0 = sg * UNIT;
      } else {  // two padded rows down, to stay positive
        qg = i * UNIT + 2 * a.pitch;
        qx = qg + (dy - 1) * a.pitch - 1;
        h0 = -2;
        w0 = -1;
      }
      auto copy = [&](const bf16* src, int cs, uint32_t to, int q, int row) {
        int h, w;
        if (a.segment) {
          h = h0 + row;
          w = w0 + q;
        } else {
          const uint32_t r = __umulhi((uint32_t)q, a.inv_pitch);
          h = h0 + (int)r;
          w = w0 + (int)(q - r * a.pitch);
        }
        const bool in = (unsigned)h < (unsigned)a.H && (unsigned)w < (unsigned)a.W;
        src += in ? (int64_t)(h * a.W + w) * cs : 0;
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(to), "l"(src),
                     "r"(in ? 16 : 0)  // 0: zero fill
                     : "memory");
      };
      {
        const int c = tid % CHX;
        const bf16* src = a.X + img * a.csx + (nt * CHX + c) * 8;
        const uint32_t to = dst + gbytes + c * XPLANE;
#pragma unroll
        for (int k = 0; k < (UNIT + 2 + 32 * CW / CHX - 1) / (32 * CW / CHX); ++k) {
          const int p = tid / CHX + k * (32 * CW / CHX);
          if (p < UNIT + 2) copy(src, a.csx, to + p * 16, qx + p, dy - 1);
        }
      }
      {  // `lanes` lanes per position, one for each plane of the gradient
        const int c = tid & (a.lanes - 1);
        const bf16* src = a.G + img * a.csg + c * 8;
        const uint32_t to = dst + c * GPLANE;
        if (c < chg)
#pragma unroll 4
          for (int p = tid >> a.lane_bits; p < UNIT; p += (32 * CW) >> a.lane_bits)
            copy(src, a.csg, to + p * 16, qg + p, 0);
      }
      asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(full_u + 8 * st)
                   : "memory");
      if (++st == a.nbuf) {
        st = 0;
        ++round;
      }
      if (++sg == seg) {
        sg = 0;
        ++hh;
      }
      if (++i == a.per_img) {
        i = hh = sg = 0;
        ++b;
      }
    }
    asm volatile("cp.async.wait_all;" ::: "memory");  // nothing in flight when the CTA ends
  } else if (warp == CW) {
    // ---------------- MMA issuer (warp-uniform, one elected lane issues)
    uint32_t leader;
    asm volatile(
        "{\n .reg .pred p;\n elect.sync _|p, 0xffffffff;\n selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(leader));
    auto commit = [&](uint32_t bar) {
      asm volatile(
          "{\n .reg .pred q;\n setp.ne.b32 q, %1, 0;\n"
          " @q tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n}\n" ::"r"(
              bar),
          "r"(leader)
          : "memory");
    };
    bool ok = true;
    int it = 0, st = 0, round = 0;
    for (int t = u0; t < u1; ++t, ++it) {
      ok = __all_sync(0xffffffffu, mbar_wait_ab(full_u + 8 * st, round & 1, abort)) != 0;
      if (!ok) break;
      // the copies' writes (generic proxy) before the MMAs' reads (async proxy)
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      tc_fence_after();
      // MN-major: the K groups (8 pixels) 128 bytes apart, the M or N groups a plane
      const uint64_t ad0 = narrow::desc_plain(buf_u + st * bufb, 128, GPLANE);
      const uint64_t bd0 = narrow::desc_plain(buf_u + st * bufb + gbytes, 128, XPLANE);
#pragma unroll
      for (int dx = 0; dx < 3; ++dx) {
#pragma unroll
        for (int kk = 0; kk < UNIT / 16; ++kk) {
          const uint64_t ad = ad0 + (uint32_t)(kk * 16), bd = bd0 + (uint32_t)(dx + kk * 16);
          asm volatile(
              "{\n .reg .pred p, q;\n setp.ne.b32 p, %4, 0;\n setp.ne.b32 q, %5, 0;\n"
              " @q tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(
                  tmem + (uint32_t)(dx * BN)),
              "l"(ad), "l"(bd), "r"(IDESC), "r"((kk > 0 || it > 0) ? 1u : 0u), "r"(leader)
              : "memory");
        }
      }
      commit(empty_u + 8 * st);
      if (++st == a.nbuf) {
        st = 0;
        ++round;
      }
    }
    if (!ok) s_abort = 1;
    commit(done_u);
    if (!mbar_wait(done_u, 0)) s_abort = 1;
  }
  __syncwarp();
  __syncthreads();
  tc_fence_after();
  if (s_abort) {
    if (tid == 0) atomicExch(&g_tc_error, 1);
  } else if (warp > CW) {
    // ---------------- the CTA's slice: row = output channel
    const int q = warp & 3, co = q * 32 + lane;
    float* out = a.partial + ((size_t)slice * a.Co + co) * 9 * a.Ci + nt * BN;
#pragma unroll 1
    for (int dx = 0; dx < 3; ++dx) {
      uint32_t v[32];
      tmem_ld32(tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(dx * BN), v);
      if (co < a.Co) {
#pragma unroll
        for (int k = 0; k < BN; k += 4)
          *reinterpret_cast<float4*>(out + (dy * 3 + dx) * a.Ci + k) =
              make_float4(__uint_as_float(v[k]), __uint_as_float(v[k + 1]),
                          __uint_as_float(v[k + 2]), __uint_as_float(v[k + 3]));
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == CW) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(COLS)
                 : "memory");
  }
}

}  // namespace wgrad
