// The collisions of two nodes at once in packed FP32 (f32x2).
//
// A packed instruction does two FP32 operations for one issue slot (its rate
// is half the scalar one, so the FP32 peak is the same: 79 TFLOP/s measured
// either way).  The scalar collision spends about two thirds of its issue slots
// on FP32 arithmetic, so packing leaves slots for the loads, stores and address
// arithmetic, which a kernel that is bound by issue is short of.
//
// Every operation is written out with its rounding: the products that are
// fused into a sum here are those the compiler fuses in collide(), found by
// comparing every intermediate moment and population bit by bit, so that the
// result is bit-identical to collide<FORCE, SM, COMP> (and collide_scaled).
// Signs are arranged so that no negation is needed: a trailing n marks the
// negative of a quantity (rounding is symmetric, so it is exact).
#pragma once

#include "ddflb_device.cuh"

namespace ddflb {

typedef float2 F2;

// 16-bit storage: two adjacent populations as one 4-byte word
template <typename S> __device__ __forceinline__ F2 widen(unsigned w);
template <> __device__ __forceinline__ F2 widen<__half>(unsigned w) {
  return __half22float2(*reinterpret_cast<const __half2*>(&w));
}
template <> __device__ __forceinline__ F2 widen<__nv_bfloat16>(unsigned w) {
  return make_float2(__uint_as_float(w << 16), __uint_as_float(w & 0xffff0000u));
}
__device__ __forceinline__ float widen1(__half v) { return __half2float(v); }
__device__ __forceinline__ float widen1(__nv_bfloat16 v) { return __bfloat162float(v); }
template <typename S> __device__ __forceinline__ unsigned narrow(F2 v);
template <> __device__ __forceinline__ unsigned narrow<__half>(F2 v) {
  const __half2 h = __floats2half2_rn(v.x, v.y);
  return *reinterpret_cast<const unsigned*>(&h);
}
template <> __device__ __forceinline__ unsigned narrow<__nv_bfloat16>(F2 v) {
  const __nv_bfloat162 h = __floats2bfloat162_rn(v.x, v.y);
  return *reinterpret_cast<const unsigned*>(&h);
}

__device__ __forceinline__ F2 add2(F2 a, F2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ F2 mul2(F2 a, F2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ F2 fma2(F2 a, F2 b, F2 c) { return __ffma2_rn(a, b, c); }

// Constants of the pair collision, each twice (the operand of a packed
// instruction is a register pair); built on the host once per context.
struct PairConst {
  struct Rates {
    F2 w1, w1n, w2, w2n, w3, w4, w4n, w5, w5n, w6, w6n, w7, w7n, w8;
  };
  Rates f, g;
  F2 rho0, rho0n, phi0, phi0n;
  F2 b1n, b2n, b1c, b1cn, b2c, b2cn;  // -beta, and beta c rounded
  F2 third, thirdn, ninth, one_n, two_n, four, eight, eight_n, half, half_n, quarter, quarter_n;
  F2 sf, isf, sg, isg;
  // body force: 1 - w/2 (c3n, c4n negated); central moments: beta - 1, 2 c
  F2 c1, c2, c3n, c4n, c5, c6, c7, c8;
  F2 b1m, b2m, c2third_n;
  F2 one, two, three, half3, half3_n, sixth, twelfth;
};

inline PairConst make_pair_const(const LbParams& P) {
  auto d = [](float v) {
    F2 r;
    r.x = v;
    r.y = v;
    return r;
  };
  auto rates = [&](const float* w) {
    return PairConst::Rates{d(w[1]), d(-w[1]), d(w[2]), d(-w[2]), d(w[3]),  d(w[4]), d(-w[4]),
                            d(w[5]), d(-w[5]), d(w[6]), d(-w[6]), d(w[7]), d(-w[7]), d(w[8])};
  };
  const float c = 1.0f / 3.0f;
  const float b1c = P.b1 * c, b2c = P.b2 * c;  // one FP32 rounding, as on the device
  PairConst K;
  K.f = rates(P.wf);
  K.g = rates(P.wg);
  K.rho0 = d(P.rho0);
  K.rho0n = d(-P.rho0);
  K.phi0 = d(P.phi0);
  K.phi0n = d(-P.phi0);
  K.b1n = d(-P.b1);
  K.b2n = d(-P.b2);
  K.b1c = d(b1c);
  K.b1cn = d(-b1c);
  K.b2c = d(b2c);
  K.b2cn = d(-b2c);
  K.third = d(c);
  K.thirdn = d(-c);
  K.ninth = d(1.0f / 9.0f);
  K.one_n = d(-1.0f);
  K.two_n = d(-2.0f);
  K.four = d(4.0f);
  K.eight = d(8.0f);
  K.eight_n = d(-8.0f);
  K.half = d(0.5f);
  K.half_n = d(-0.5f);
  K.quarter = d(0.25f);
  K.quarter_n = d(-0.25f);
  K.sf = d(P.sf);
  K.isf = d(P.isf);
  K.sg = d(P.sg);
  K.isg = d(P.isg);
  auto c_of = [&](int k) { return 1.0f - 0.5f * P.wf[k]; };  // (0.5 w is exact)
  K.c1 = d(c_of(1));
  K.c2 = d(c_of(2));
  K.c3n = d(-c_of(3));
  K.c4n = d(-c_of(4));
  K.c5 = d(c_of(5));
  K.c6 = d(c_of(6));
  K.c7 = d(c_of(7));
  K.c8 = d(c_of(8));
  K.b1m = d(P.b1 - 1.0f);
  K.b2m = d(P.b2 - 1.0f);
  K.c2third_n = d(-2.0f * c);
  K.one = d(1.0f);
  K.two = d(2.0f);
  K.three = d(3.0f);
  K.half3 = d(1.5f);
  K.half3_n = d(-1.5f);
  K.sixth = d(1.0f / 6.0f);
  K.twelfth = d(1.0f / 12.0f);
  return K;
}

__device__ __forceinline__ F2 sub2(F2 a, F2 b) {
  return __fadd2_rn(a, make_float2(-b.x, -b.y));  // (a source modifier)
}

struct Ef2 {
  F2 s, e;
};
__device__ __forceinline__ Ef2 two_sum2(F2 a, F2 b) {
  const F2 s = add2(a, b), bb = sub2(s, a);
  return Ef2{s, add2(sub2(a, sub2(s, bb)), sub2(b, bb))};
}
__device__ __forceinline__ Ef2 two_diff2(F2 a, F2 b) {
  const F2 s = sub2(a, b), bb = sub2(s, a);
  return Ef2{s, sub2(sub2(a, sub2(s, bb)), add2(b, bb))};
}

// the relaxation of relax() from the non-equilibrium moments; n5n .. n8n are
// negatives (w6, w6n, w7, w7n swapped by the caller where n6, n7 are not)
template <bool N12>
__device__ __forceinline__ void relax2(const PairConst& K, const PairConst::Rates& w, F2 w6, F2 w6n,
                                       F2 w7, F2 w7n, F2 n1, F2 n2, F2 n3, F2 n4, F2 n5n, F2 n6n,
                                       F2 n7n, F2 n8n, F2 d[9]) {
  const F2 d3 = mul2(w.w3, n3), d8n = mul2(w.w8, n8n);
  const F2 xx = mul2(K.half, fma2(w.w4, n4, d3)), yy = mul2(K.half, fma2(w.w4n, n4, d3));
  d[0] = add2(d[0], fma2(w.w8, n8n, d3));
  const F2 xp = N12 ? fma2(w.w1, n1, xx) : xx, yp = N12 ? fma2(w.w2, n2, yy) : yy;
  const F2 xm = N12 ? fma2(w.w1n, n1, xx) : xx, ym = N12 ? fma2(w.w2n, n2, yy) : yy;
  d[1] = fma2(K.half_n, fma2(w.w8, n8n, fma2(w7, n7n, xp)), d[1]);
  d[2] = fma2(K.half_n, fma2(w.w8, n8n, fma2(w6, n6n, yp)), d[2]);
  d[3] = fma2(K.half_n, fma2(w.w8, n8n, fma2(w7n, n7n, xm)), d[3]);
  d[4] = fma2(K.half_n, fma2(w.w8, n8n, fma2(w6n, n6n, ym)), d[4]);
  const F2 pn = fma2(w.w5, n5n, d8n), qn = fma2(w6, n6n, mul2(w7, n7n));
  const F2 rn = fma2(w.w5n, n5n, d8n), sn = fma2(w6, n6n, mul2(w7n, n7n));
  d[5] = fma2(K.quarter, add2(pn, qn), d[5]);
  d[6] = fma2(K.quarter, add2(rn, sn), d[6]);
  d[7] = fma2(K.quarter, sub2(pn, qn), d[7]);
  d[8] = fma2(K.quarter, sub2(rn, sn), d[8]);
}

// k b - a with the product split exactly: the negative of sub_scaled()
__device__ __forceinline__ F2 sub_scaled2n(const Ef2& a, F2 k, F2 kn,
                                           const Ef2& b) {
  const F2 p = mul2(k, b.s), pen = fma2(kn, b.s, p);
  const F2 t = fma2(kn, b.e, add2(a.e, pen));
  return sub2(sub2(p, a.s), t);
}

// cross_diff() for the constants ka, kb
__device__ __forceinline__ F2 cross_diff2(F2 ka, F2 kan, const Ef2& a, F2 kb,
                                          F2 kbn, const Ef2& b) {
  const F2 p = mul2(ka, a.s), pen = fma2(kan, a.s, p);
  const F2 r = mul2(kb, b.s), ren = fma2(kbn, b.s, r);
  const F2 m = fma2(ka, a.e, mul2(kbn, b.e));
  return add2(sub2(p, r), add2(sub2(ren, pen), m));
}

// relax_source(): n5n .. n8n are negatives; Fx, Fy the force of each node
__device__ __forceinline__ void relax_source2(const PairConst& K, F2 ux, F2 uy, F2 Fx, F2 Fy, F2 w6,
                                              F2 w7, F2 n3, F2 n4, F2 n5n, F2 n6, F2 n7, F2 n8n,
                                              F2 d[9]) {
  const PairConst::Rates& w = K.f;
  // source()
  const F2 sxx = mul2(mul2(K.two, Fx), ux), syy = mul2(mul2(K.two, Fy), uy);
  const F2 fxuy = mul2(Fx, uy), fyux = mul2(Fy, ux);
  const F2 s6 = fma2(fyux, ux, mul2(sxx, uy)), s7 = fma2(fxuy, uy, mul2(syy, ux));
  const F2 s8 =
      mul2(K.two, fma2(mul2(mul2(Fx, ux), uy), uy, mul2(mul2(mul2(Fy, uy), ux), ux)));
  const F2 D1n = mul2(K.c1, Fx), D2n = mul2(K.c2, Fy);
  const F2 D3 = fma2(w.w3, n3, mul2(K.c3n, add2(sxx, syy)));
  const F2 D4 = fma2(w.w4, n4, mul2(K.c4n, sub2(sxx, syy)));
  const F2 D5n = fma2(w.w5, n5n, mul2(K.c5, add2(fxuy, fyux)));
  const F2 D6n = fma2(w6, n6, mul2(K.c6, s6)), D7n = fma2(w7, n7, mul2(K.c7, s7));
  const F2 D8n = fma2(w.w8, n8n, mul2(K.c8, s8));
  const F2 xx = mul2(K.half, add2(D3, D4)), yy = mul2(K.half, sub2(D3, D4));
  d[0] = add2(d[0], add2(D3, D8n));
  d[1] = fma2(K.half_n, add2(add2(sub2(xx, D1n), D7n), D8n), d[1]);
  d[2] = fma2(K.half_n, add2(add2(sub2(yy, D2n), D6n), D8n), d[2]);
  d[3] = fma2(K.half_n, add2(sub2(add2(D1n, xx), D7n), D8n), d[3]);
  d[4] = fma2(K.half_n, add2(sub2(add2(D2n, yy), D6n), D8n), d[4]);
  const F2 pn = add2(D5n, D8n), qn = add2(D6n, D7n), rn = sub2(D8n, D5n), sn = sub2(D6n, D7n);
  d[5] = fma2(K.quarter, add2(pn, qn), d[5]);
  d[6] = fma2(K.quarter, add2(rn, sn), d[6]);
  d[7] = fma2(K.quarter, sub2(pn, qn), d[7]);
  d[8] = fma2(K.quarter, sub2(rn, sn), d[8]);
}

// central_neq() and relax_cascaded() (SM 2) or relax_central() (SM 3) from the
// scalar lattice's raw non-equilibrium moments
template <int SM>
__device__ __forceinline__ void relax_cm2(const PairConst& K, F2 ux, F2 uy, F2 uxx, F2 uyy, F2 phi,
                                          F2 rx, F2 ry, F2 n3, F2 n4, F2 rxy, F2 rxxy, F2 rxyy,
                                          F2 n8, F2 d[9]) {
  const PairConst::Rates& w = K.g;
  const F2 ux2 = mul2(K.two, ux), uy2 = mul2(K.two, uy);
  const F2 ux2n = mul2(K.two_n, ux), uy2n = mul2(K.two_n, uy);
  const F2 p = mul2(ux, uy), p2 = mul2(K.two, p), p4 = mul2(K.four, p);
  F2 vx, vy, vxy, vxxy, vxyy, vxxyy, vs, vd;
  {
    const F2 rxx = mul2(K.half, add2(n3, n4)), ryy = mul2(K.half, sub2(n3, n4));
    const F2 uxn = mul2(ux, K.one_n), uyn = mul2(uy, K.one_n);
    vx = rx;
    vy = ry;
    const F2 vxx = fma2(ux2n, rx, rxx), vyy = fma2(uy2n, ry, ryy);
    vs = add2(vxx, vyy);
    vd = sub2(vxx, vyy);
    vxy = fma2(uxn, ry, fma2(uyn, rx, rxy));
    vxxy = fma2(p2, rx, fma2(uyn, rxx, fma2(uxx, ry, fma2(ux2n, rxy, rxxy))));
    vxyy = fma2(p2, ry, fma2(uxn, ryy, fma2(uyy, rx, fma2(uy2n, rxy, rxyy))));
    const F2 in = fma2(mul2(K.b2m, ux), ux, mul2(mul2(K.b1m, uy), uy));
    F2 t = fma2(mul2(K.c2third_n, phi), in, n8);
    t = fma2(uy2n, rxxy, fma2(ux2n, rxyy, t));
    t = fma2(p4, rxy, fma2(uyy, rxx, fma2(uxx, ryy, t)));
    vxxyy = fma2(mul2(p, uy2n), rx, fma2(mul2(uxx, uy2n), ry, t));
  }
  if (SM == 2) {
    const F2 h1 = mul2(mul2(w.w1n, vx), K.sixth), h2 = mul2(mul2(w.w2n, vy), K.sixth);
    const F2 uyh2 = mul2(uy, h2);
    const F2 h3 = fma2(mul2(mul2(w.w3, K.one_n), vs), K.twelfth, fma2(ux, h1, uyh2));
    const F2 h4 = fma2(K.three, fma2(ux, h1, mul2(uyh2, K.one_n)),
                       mul2(mul2(w.w4n, vd), K.quarter));
    const F2 h5 = fma2(K.half3, fma2(uy, h1, mul2(ux, h2)), mul2(mul2(w.w5n, vxy), K.quarter));
    const F2 p3 = mul2(mul2(K.three, ux), uy);
    F2 t = fma2(mul2(w.w6, vxxy), K.quarter, mul2(ux2n, h5));
    t = fma2(mul2(K.half_n, uy), h4, t);
    t = fma2(mul2(K.half3_n, uy), h3, t);
    t = fma2(fma2(K.half3, uxx, K.one), h2, t);
    const F2 h6 = fma2(p3, h1, t);
    t = fma2(mul2(w.w7, vxyy), K.quarter, mul2(uy2n, h5));
    t = fma2(mul2(K.half, ux), h4, t);
    t = fma2(mul2(K.half3_n, ux), h3, t);
    t = fma2(p3, h2, t);
    const F2 h7 = fma2(fma2(K.half3, uyy, K.one), h1, t);
    t = fma2(mul2(mul2(w.w8, K.one_n), vxxyy), K.quarter, mul2(ux2n, h7));
    t = fma2(uy2n, h6, t);
    t = fma2(mul2(p4, K.one_n), h5, t);
    t = fma2(mul2(K.half, sub2(uxx, uyy)), h4, t);
    t = fma2(fma2(K.half3_n, add2(uxx, uyy), K.two_n), h3, t);
    t = fma2(mul2(fma2(K.three, uxx, K.two), uy), h2, t);
    const F2 h8 = fma2(mul2(fma2(K.three, uyy, K.two), ux), h1, t);
    d[0] = fma2(K.four, sub2(h8, h3), d[0]);
    const F2 a13 = add2(h1, h3), a23 = add2(h2, h3), s12 = add2(h1, h2), e12 = sub2(h1, h2);
    d[1] = add2(d[1], fma2(K.two_n, h8, fma2(K.two, h7, add2(sub2(h1, h3), h4))));
    d[2] = add2(d[2], fma2(K.two_n, h8, fma2(K.two, h6, sub2(sub2(h2, h3), h4))));
    d[3] = add2(d[3], fma2(K.two_n, h8, fma2(K.two_n, h7, sub2(h4, a13))));
    d[4] = sub2(d[4], fma2(K.two, h8, fma2(K.two, h6, add2(a23, h4))));
    const F2 h32 = mul2(K.two, h3);
    d[5] = add2(d[5], add2(sub2(sub2(add2(add2(s12, h32), h5), h6), h7), h8));
    d[6] = add2(d[6], add2(add2(sub2(sub2(sub2(h32, e12), h5), h6), h7), h8));
    d[7] = add2(d[7], add2(add2(add2(add2(sub2(h32, s12), h5), h6), h7), h8));
    d[8] = add2(d[8], add2(sub2(add2(sub2(add2(e12, h32), h5), h6), h7), h8));
  } else {
    const F2 w3n = mul2(w.w3, K.one_n);
    const F2 Dx = mul2(w.w1n, vx), Dy = mul2(w.w2n, vy);
    const F2 Dxx = mul2(K.half, fma2(w3n, vs, mul2(w.w4n, vd)));
    const F2 Dyy = mul2(K.half, fma2(w3n, vs, mul2(w.w4, vd)));
    const F2 Dxy = mul2(w.w5n, vxy), Dxxy = mul2(w.w6n, vxxy), Dxyy = mul2(w.w7n, vxyy);
    const F2 Dxxyy = mul2(mul2(w.w8, K.one_n), vxxyy);
    const F2 Rxx = fma2(ux2, Dx, Dxx), Ryy = fma2(uy2, Dy, Dyy);
    const F2 Rxy = fma2(ux, Dy, fma2(uy, Dx, Dxy));
    const F2 Rxxy = fma2(p2, Dx, fma2(uy, Dxx, fma2(uxx, Dy, fma2(ux2, Dxy, Dxxy))));
    const F2 Rxyy = fma2(p2, Dy, fma2(ux, Dyy, fma2(uyy, Dx, fma2(uy2, Dxy, Dxyy))));
    F2 R4 = fma2(uy2, Dxxy, fma2(ux2, Dxyy, Dxxyy));
    R4 = fma2(p4, Dxy, fma2(uyy, Dxx, fma2(uxx, Dyy, R4)));
    R4 = fma2(mul2(p, uy2), Dx, fma2(mul2(uxx, uy2), Dy, R4));
    // populations()
    const F2 m3 = add2(Rxx, Ryy), m4 = sub2(Rxx, Ryy);
    const F2 kxx = mul2(K.half, add2(m3, m4)), kyy = mul2(K.half, sub2(m3, m4));
    d[0] = add2(d[0], sub2(R4, m3));
    d[1] = fma2(K.half, sub2(sub2(add2(Dx, kxx), Rxyy), R4), d[1]);
    d[2] = fma2(K.half, sub2(sub2(add2(Dy, kyy), Rxxy), R4), d[2]);
    d[3] = fma2(K.half, sub2(add2(sub2(kxx, Dx), Rxyy), R4), d[3]);
    d[4] = fma2(K.half, sub2(add2(sub2(kyy, Dy), Rxxy), R4), d[4]);
    const F2 a = add2(Rxy, R4), b = add2(Rxxy, Rxyy), r = sub2(R4, Rxy), e = sub2(Rxxy, Rxyy);
    d[5] = fma2(K.quarter, add2(a, b), d[5]);
    d[6] = fma2(K.quarter, add2(r, e), d[6]);
    d[7] = fma2(K.quarter, sub2(a, b), d[7]);
    d[8] = fma2(K.quarter, sub2(r, e), d[8]);
  }
}

// Both collisions of two nodes.  COMP: FP32 storage, deviations, compensated
// odd moments; otherwise populations in storage units (as collide_scaled()),
// or in physical ones with a force (Fx, Fy at the two nodes) or SM 2 or 3.
template <bool COMP, bool FORCE = false, int SM = 0>
__device__ __forceinline__ void collide_pair(const PairConst& K, F2 f[9], F2 g[9],
                                             F2 Fx = F2{}, F2 Fy = F2{}) {
  constexpr bool PHYS = COMP || FORCE || SM != 0;
  // ---- flow moments
  const F2 s57 = add2(f[5], f[7]), s68 = add2(f[6], f[8]);
  const F2 fkxyn = sub2(s68, s57);
  const F2 s13 = add2(f[1], f[3]), s24 = add2(f[2], f[4]);
  const F2 fm4 = sub2(s13, s24), A = add2(s13, s24), B = add2(s57, s68);
  const F2 T3 = fma2(K.two_n, f[0], fma2(K.four, B, A));
  const F2 T8n = add2(fma2(K.eight_n, B, A), f[0]);
  const F2 fk0 = add2(f[0], add2(A, B));
  Ef2 ofx, ofy, ofxxy, ofxyy;
  if (COMP) {
    const Ef2 a57 = two_diff2(f[5], f[7]), a68 = two_diff2(f[6], f[8]);
    const Ef2 d13 = two_diff2(f[1], f[3]), d24 = two_diff2(f[2], f[4]);
    ofxxy = two_sum2(a57.s, a68.s);
    ofxxy.e = add2(ofxxy.e, add2(a57.e, a68.e));
    ofxyy = two_diff2(a57.s, a68.s);
    ofxyy.e = add2(ofxyy.e, sub2(a57.e, a68.e));
    ofx = two_sum2(d13.s, ofxyy.s);
    ofx.e = add2(ofx.e, add2(d13.e, ofxyy.e));
    ofy = two_sum2(d24.s, ofxxy.s);
    ofy.e = add2(ofy.e, add2(d24.e, ofxxy.e));
  } else {
    const F2 a57 = sub2(f[5], f[7]), a68 = sub2(f[6], f[8]);
    ofxxy.s = add2(a57, a68);
    ofxyy.s = sub2(a57, a68);
    ofx.s = add2(sub2(f[1], f[3]), ofxyy.s);
    ofy.s = add2(sub2(f[2], f[4]), ofxxy.s);
  }
  if (FORCE) {  // the half-force momentum shift, exactly where compensated
    const F2 hx = mul2(K.half, Fx), hy = mul2(K.half, Fy);
    if (COMP) {
      const Ef2 sx = two_sum2(ofx.s, hx), sy = two_sum2(ofy.s, hy);
      ofx = Ef2{sx.s, add2(sx.e, ofx.e)};
      ofy = Ef2{sy.s, add2(sy.e, ofy.e)};
    } else {
      ofx.s = add2(ofx.s, hx);
      ofy.s = add2(ofy.s, hy);
    }
  }
  const F2 fkx = ofx.s, fky = ofy.s;
  // ---- scalar moments
  const F2 qn = mul2(K.quarter_n, g[0]);
  const F2 gkxyn = add2(sub2(g[6], g[5]), sub2(g[8], g[7]));
  const F2 gm4 = add2(sub2(g[1], g[2]), sub2(g[3], g[4]));
  const F2 t1 = add2(add2(add2(g[1], qn), add2(g[3], qn)), add2(add2(g[2], qn), add2(g[4], qn)));
  const F2 t2 = add2(add2(fma2(K.four, g[5], qn), fma2(K.four, g[7], qn)),
                     add2(fma2(K.four, g[6], qn), fma2(K.four, g[8], qn)));
  const F2 G3 = add2(t1, t2);
  const F2 G8n =
      add2(add2(sub2(g[1], fma2(K.eight, g[5], qn)), sub2(g[3], fma2(K.eight, g[7], qn))),
           add2(sub2(g[2], fma2(K.eight, g[6], qn)), sub2(g[4], fma2(K.eight, g[8], qn))));
  const F2 gk0 = add2(add2(g[0], add2(add2(g[1], g[3]), add2(g[2], g[4]))),
                      add2(add2(g[5], g[7]), add2(g[6], g[8])));
  // ---- macroscopic state (physical units)
  const F2 dr = PHYS ? fk0 : mul2(fk0, K.isf), dp = PHYS ? gk0 : mul2(gk0, K.isg);
  const F2 ukx = PHYS ? fkx : mul2(fkx, K.isf), uky = PHYS ? fky : mul2(fky, K.isf);
  const F2 rho = add2(K.rho0, dr);
  F2 irho;
  irho.x = __frcp_rn(rho.x);
  irho.y = __frcp_rn(rho.y);
  const F2 ux = mul2(ukx, irho), uy = mul2(uky, irho);
  const F2 uxx = mul2(ux, ux), uyy = mul2(uy, uy), usq = add2(uxx, uyy);
  const F2 difn = sub2(uyy, uxx);
  const F2 X = fma2(uxx, uyy, mul2(K.third, usq));
  const F2 phi = add2(K.phi0, dp);
  // rho and phi in the units of the populations
  const F2 rs = PHYS ? rho : mul2(rho, K.sf), ps = PHYS ? phi : mul2(phi, K.sg);
  const F2 rsn = mul2(rs, K.one_n), psn = mul2(ps, K.one_n);
  // ---- flow
  {
    const F2 n3 = fma2(T3, K.third, mul2(rsn, usq)), n4 = fma2(rs, difn, fm4);
    const F2 n5n = fma2(fkx, uy, fkxyn), n8n = fma2(T8n, K.ninth, mul2(rs, X));
    const F2 z = K.one_n;  // (unused: the flow's first moments are conserved)
    if (COMP) {
      const F2 n6n = fma2(fky, uxx, sub_scaled2n(ofxxy, K.third, K.thirdn, ofy));
      const F2 n7n = fma2(fkx, uyy, sub_scaled2n(ofxyy, K.third, K.thirdn, ofx));
      if (FORCE)
        relax_source2(K, ux, uy, Fx, Fy, K.f.w6, K.f.w7, n3, n4, n5n, n6n, n7n, n8n, f);
      else
        relax2<false>(K, K.f, K.f.w6, K.f.w6n, K.f.w7, K.f.w7n, z, z, n3, n4, n5n, n6n, n7n, n8n, f);
    } else {
      const F2 n6 = fma2(fky, sub2(K.thirdn, uxx), ofxxy.s);
      const F2 n7 = fma2(fkx, sub2(K.thirdn, uyy), ofxyy.s);
      if (FORCE)
        relax_source2(K, ux, uy, Fx, Fy, K.f.w6n, K.f.w7n, n3, n4, n5n, n6, n7, n8n, f);
      else
        relax2<false>(K, K.f, K.f.w6n, K.f.w6, K.f.w7n, K.f.w7, z, z, n3, n4, n5n, n6, n7, n8n, f);
    }
  }
  // ---- scalar
  const F2 n3 = fma2(G3, K.third, mul2(psn, usq)), n4 = fma2(ps, difn, gm4);
  const F2 n5n = fma2(mul2(ps, ux), uy, gkxyn), n8n = fma2(G8n, K.ninth, mul2(ps, X));
  if (COMP) {
    const Ef2 a57 = two_diff2(g[5], g[7]), a68 = two_diff2(g[6], g[8]);
    const Ef2 d13 = two_diff2(g[1], g[3]), d24 = two_diff2(g[2], g[4]);
    Ef2 xxy = two_sum2(a57.s, a68.s);
    xxy.e = add2(xxy.e, add2(a57.e, a68.e));
    Ef2 xyy = two_diff2(a57.s, a68.s);
    xyy.e = add2(xyy.e, sub2(a57.e, a68.e));
    Ef2 x = two_sum2(d13.s, xyy.s);
    x.e = add2(x.e, add2(d13.e, xyy.e));
    Ef2 y = two_sum2(d24.s, xxy.s);
    y.e = add2(y.e, add2(d24.e, xxy.e));
    const F2 dpn = mul2(dp, K.one_n);
    const F2 n1 = mul2(add2(cross_diff2(K.rho0, K.rho0n, x, K.phi0, K.phi0n, ofx),
                            fma2(x.s, dr, mul2(dpn, fkx))), irho);
    const F2 n2 = mul2(add2(cross_diff2(K.rho0, K.rho0n, y, K.phi0, K.phi0n, ofy),
                            fma2(y.s, dr, mul2(dpn, fky))), irho);
    const F2 px = sub2(x.s, n1), py = sub2(y.s, n2);
    const F2 n6n = fma2(py, uxx, fma2(K.b1cn, n2, sub_scaled2n(xxy, K.b1c, K.b1cn, y)));
    const F2 n7n = fma2(px, uyy, fma2(K.b2cn, n1, sub_scaled2n(xyy, K.b2c, K.b2cn, x)));
    if constexpr (SM == 0)
      relax2<true>(K, K.g, K.g.w6, K.g.w6n, K.g.w7, K.g.w7n, n1, n2, n3, n4, n5n, n6n, n7n, n8n, g);
    else
      relax_cm2<SM>(K, ux, uy, uxx, uyy, phi, n1, n2, n3, n4, mul2(n5n, K.one_n),
                    mul2(n6n, K.one_n), mul2(n7n, K.one_n), mul2(n8n, K.one_n), g);
  } else {
    const F2 a57 = sub2(g[5], g[7]), a68 = sub2(g[6], g[8]);
    const F2 kxxy = add2(a57, a68), kxyy = sub2(a57, a68);
    const F2 kx = add2(sub2(g[1], g[3]), kxyy), ky = add2(sub2(g[2], g[4]), kxxy);
    const F2 txn = mul2(psn, ukx), ex = fma2(ps, ukx, txn);
    const F2 tyn = mul2(psn, uky), ey = fma2(ps, uky, tyn);
    const F2 n1 = mul2(sub2(fma2(kx, rho, txn), ex), irho);
    const F2 n2 = mul2(sub2(fma2(ky, rho, tyn), ey), irho);
    // -(beta c + u^2): the product fused, as the compiler does with one use
    const F2 e6n = fma2(K.b1n, K.third, mul2(uxx, K.one_n));
    const F2 e7n = fma2(K.b2n, K.third, mul2(uyy, K.one_n));
    const F2 n6 = fma2(mul2(ps, uy), e6n, kxxy), n7 = fma2(mul2(ps, ux), e7n, kxyy);
    if constexpr (SM == 0)
      relax2<true>(K, K.g, K.g.w6n, K.g.w6, K.g.w7n, K.g.w7, n1, n2, n3, n4, n5n, n6, n7, n8n, g);
    else
      relax_cm2<SM>(K, ux, uy, uxx, uyy, phi, n1, n2, n3, n4, mul2(n5n, K.one_n), n6, n7,
                    mul2(n8n, K.one_n), g);
  }
}

}  // namespace ddflb
