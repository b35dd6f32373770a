// lb_collide.cuh -- the D3Q19 collision of Eq. 5 (BGK relaxation to the Eq. 6
// equilibrium, body-force source, optional thermal source F_p) and the update
// of one node (pull streaming + collision + store), shared by the
// stream-collide kernels.
#pragma once

#include "lb_pull.cuh"

namespace lbmd {

constexpr int kRowsPerBlock = 8;  // block = 32 x 8 threads

// Weight-orthogonal D3Q19 mode basis, row k at velocity c_p:
// 0: 1; 1-3: c_x, c_y, c_z; 4: c^2 - 1; 5: 3c_x^2 - c^2; 6: c_y^2 - c_z^2;
// 7-9: c_x c_y, c_y c_z, c_z c_x; 10-12: (3c^2 - 5) c_x, c_y, c_z;
// 13: (c_y^2 - c_z^2) c_x; 14: (c_z^2 - c_x^2) c_y; 15: (c_x^2 - c_y^2) c_z;
// 16: 3c^4 - 6c^2 + 1; 17: (2c^2 - 3)(3c_x^2 - c^2); 18: (2c^2 - 3)(c_y^2 - c_z^2).
__host__ __device__ constexpr int mode_row(int k, int p) {
  const int x = cx(p), y = cy(p), z = cz(p), c2 = x * x + y * y + z * z;
  return k == 0 ? 1 : k == 1 ? x : k == 2 ? y : k == 3 ? z
       : k == 4 ? c2 - 1 : k == 5 ? 3 * x * x - c2 : k == 6 ? y * y - z * z
       : k == 7 ? x * y : k == 8 ? y * z : k == 9 ? z * x
       : k == 10 ? (3 * c2 - 5) * x : k == 11 ? (3 * c2 - 5) * y : k == 12 ? (3 * c2 - 5) * z
       : k == 13 ? (y * y - z * z) * x : k == 14 ? (z * z - x * x) * y
       : k == 15 ? (x * x - y * y) * z : k == 16 ? 3 * c2 * c2 - 6 * c2 + 1
       : k == 17 ? (2 * c2 - 3) * (3 * x * x - c2) : (2 * c2 - 3) * (y * y - z * z);
}

// Arithmetic of the collision, on one node (Ops1: float) or on two nodes at
// once (Ops2: float2, the paired FP32 instructions of sm_100 and later).  A
// paired operation is two independent correctly rounded operations, so both
// give the same bits for the same node.  Every operation is written out with
// its rounding (no contraction left to the compiler), so every stream-collide
// kernel -- pull, in-place, ensemble, one or two nodes per thread -- rounds
// identically.
struct Ops1 {
  using V = float;
  static constexpr int N = 1;  // nodes
  static __device__ __forceinline__ V pack(const float *v) { return v[0]; }
  static __device__ __forceinline__ void unpack(V v, float *o) { o[0] = v; }
  static __device__ __forceinline__ V add(V a, V b) { return __fadd_rn(a, b); }
  static __device__ __forceinline__ V sub(V a, V b) { return __fadd_rn(a, -b); }
  static __device__ __forceinline__ V mul(V a, V b) { return __fmul_rn(a, b); }
  static __device__ __forceinline__ V fma(V a, V b, V c) { return fmaf(a, b, c); }
  static __device__ __forceinline__ V neg(V a) { return -a; }
  static __device__ __forceinline__ V splat(float s) { return s; }
  static __device__ __forceinline__ V rcp(V a) { return __frcp_rn(a); }  // as 1.0f / a
  static __device__ __forceinline__ bool finite(V a) { return isfinite(a); }
};
struct Ops2 {
  using V = float2;
  static constexpr int N = 2;
  static __device__ __forceinline__ V pack(const float *v) { return make_float2(v[0], v[1]); }
  static __device__ __forceinline__ void unpack(V v, float *o) {
    o[0] = v.x;
    o[1] = v.y;
  }
  static __device__ __forceinline__ V neg(V a) { return make_float2(-a.x, -a.y); }
  static __device__ __forceinline__ V add(V a, V b) { return __fadd2_rn(a, b); }
  static __device__ __forceinline__ V sub(V a, V b) { return __fadd2_rn(a, neg(b)); }
  static __device__ __forceinline__ V mul(V a, V b) { return __fmul2_rn(a, b); }
  static __device__ __forceinline__ V fma(V a, V b, V c) { return __ffma2_rn(a, b, c); }
  static __device__ __forceinline__ V splat(float s) { return make_float2(s, s); }
  static __device__ __forceinline__ V rcp(V a) { return make_float2(__frcp_rn(a.x), __frcp_rn(a.y)); }
  static __device__ __forceinline__ bool finite(V a) { return isfinite(a.x) && isfinite(a.y); }
};

// Uniforms (k + 1/2) 2^-23 in (0, 1), as uniform23 gives them: 1 + k 2^-23 by its
// bits, less 1 - 2^-24, both exact.
template <class O>
__device__ __forceinline__ typename O::V uniform23_t(const uint32_t *x) {
  float f[O::N];
#pragma unroll
  for (int n = 0; n < O::N; ++n) f[n] = __uint_as_float((x[n] >> 9) | 0x3f800000u);
  return O::add(O::pack(f), O::splat(-0.99999994f));
}

// Two standard normals per node by Box and Muller, sqrt(-2 ln u1) times the
// cosine and sine of 2 pi u2, on operations that take one or two nodes at once
// (the library functions take one, and were two fifths of the kernel).
//   ln u = e ln 2 + ln(1 + f), 2^e (1 + f) = u, sqrt(1/2) <= 1 + f < sqrt(2):
//     f - f^2/2 + f^3 Q(f), Q of degree 7 (6e-9);
//   the angle is reduced to +-pi/4 exactly (2 u2 less a multiple of 1/2), sine
//     and cosine there by polynomials in r^2 (3.1e-9, 6e-11);
//   the root from the hardware's reciprocal root and one Newton step.
// The polynomials are weighted minimax ones by Lawson's iteration, fitted again
// with their weights and errors by a test (test_noise_polynomials.py).  Against
// 64 bits over all 2^23 values of u1 and of u2: rms 4.49e-8 relative for the
// normals, largest error 1.78e-7 of the radius (library functions 4.60e-8,
// 1.77e-7).
template <class O>
__device__ __forceinline__ void box_muller_t(typename O::V u1, typename O::V u2, typename O::V &n1,
                                             typename O::V &n2) {
  using V = typename O::V;
  float u[O::N], m[O::N], ef[O::N];
  O::unpack(u1, u);
#pragma unroll
  for (int n = 0; n < O::N; ++n) {
    // k >> 23 = 64 + e: less sqrt(1/2)'s bits
    const uint32_t i = __float_as_uint(u[n]) + 0x20000000u, k = i - 0x3f3504f3u;
    m[n] = __uint_as_float(i - (k & 0xff800000u));
    ef[n] = __uint_as_float(0x4b400000u | (k >> 23));  // 1.5 2^23 + 64 + e
  }
  const V e = O::add(O::pack(ef), O::splat(-12582976.0f));
  const V f = O::add(O::pack(m), O::splat(-1.0f));
  V q = O::splat(-0.07634429633617401f);
  q = O::fma(q, f, O::splat(0.12761549651622772f));
  q = O::fma(q, f, O::splat(-0.131601944565773f));
  q = O::fma(q, f, O::splat(0.14201761782169342f));
  q = O::fma(q, f, O::splat(-0.16623356938362122f));
  q = O::fma(q, f, O::splat(0.20001226663589478f));
  q = O::fma(q, f, O::splat(-0.250008225440979f));
  q = O::fma(q, f, O::splat(0.3333333134651184f));
  q = O::mul(f, O::fma(q, f, O::splat(-0.5f)));  // ln(1 + f) = f + f (f (Q f - 1/2))
  q = O::fma(e, O::splat(-2.1219444e-4f), O::fma(f, q, f));  // ln 2 = 0.693359375 - 2.12e-4
  const V L = O::mul(O::splat(-2.0f), O::fma(e, O::splat(0.693359375f), q));
  float l[O::N];
  O::unpack(L, l);
#pragma unroll
  for (int n = 0; n < O::N; ++n) asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(l[n]) : "f"(l[n]));
  const V y = O::pack(l), s0 = O::mul(L, y);
  const V rad = O::fma(O::mul(O::splat(0.5f), y), O::fma(O::neg(s0), s0, L), s0);
  const V t = O::fma(u2, O::splat(4.0f), O::splat(12582912.0f));  // quadrant in its low bits
  const V r = O::fma(O::add(t, O::splat(-12582912.0f)), O::splat(-0.5f), O::add(u2, u2));
  const V r2 = O::mul(r, r);
  V s = O::fma(r2, O::splat(-0.5890786647796631f), O::splat(2.549767255783081f));
  s = O::fma(r2, s, O::splat(-5.167707920074463f));
  // the leading coefficient in two parts, the large one in the last, once rounded operation
  s = O::fma(O::splat(3.1415927410125732f), r, O::mul(r, O::fma(r2, s, O::splat(-9.707896709e-08f))));
  V c = O::fma(r2, O::splat(0.23142953217029572f), O::splat(-1.3350584506988525f));
  c = O::fma(r2, c, O::splat(4.0587077140808105f));
  c = O::fma(r2, c, O::splat(-4.934802055358887f));
  c = O::fma(r2, c, O::splat(1.0f));
  float k[O::N], sn[O::N], cs[O::N];
  O::unpack(t, k);
  O::unpack(s, sn);
  O::unpack(c, cs);
#pragma unroll
  for (int n = 0; n < O::N; ++n) {
    const int a = __float_as_int(k[n]);
    const float v = (a & 1) ? cs[n] : sn[n], w = (a & 1) ? sn[n] : cs[n];
    sn[n] = __int_as_float(__float_as_int(v) ^ ((a & 2) << 30));
    cs[n] = __int_as_float(__float_as_int(w) ^ (((a + 1) & 2) << 30));
  }
  n1 = O::mul(rad, O::pack(cs));
  n2 = O::mul(rad, O::pack(sn));
}

// Thermal source F_p of Eq. 5 (fluctuating LB, Adhikari et al. 2005, in the
// mode form of Duenweg, Schiller and Ladd 2007) at the nodes `node`, density
// rho:
//   xi_p = w_p sum_{k=4}^{18} e_kp a_k sqrt(rho) r_k,
//   a_k = sqrt((kT / c_s^2) (1 - (1 - omega)^2) / b_k)   (ph.fl_amp[k - 4]),
// with fifteen standard normals r_k from Box-Muller on four Philox blocks,
// counter (node, step lo, step hi, block | 2 << 8), key (seed lo, seed hi).
// The noise touches only non-conserved modes: mass and momentum are exact.
//
// Two forms, equal up to the rounding of single precision (2e-8 of the
// populations), of which launch_lb_*_fluct choose:
//  kNoiseNode: the library's logarithm, sine and cosine and a sum over all
//   modes, a node at a time;
//  kNoisePair: box_muller_t and the modes by parity, one or two nodes.
// What is rounded to 16 bits afterwards, or moves a chain, keeps kNoiseNode: a
// last bit there turns a rounding of a stored population, and after 16 steps
// the velocity field of a bfloat16 box is 1e-3 from that of the other form.
enum Noise { kNoNoise = 0, kNoiseNode = 1, kNoisePair = 2 };

__device__ __forceinline__ void thermal_source(const LbPhys &ph, uint32_t node, float rho,
                                               float xi[kQ]) {
  const long long step = *ph.step;
  float r[16];
#pragma unroll
  for (uint32_t j = 0; j < 4; ++j) {
    const U4 c{node, (uint32_t)(unsigned long long)step, (uint32_t)((unsigned long long)step >> 32),
               j | (2u << 8)};
    const U4 x = philox4x32_10(c, (uint32_t)ph.seed, (uint32_t)(ph.seed >> 32));
    const uint32_t xs[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const float rad = sqrtf(-2.0f * logf(uniform23(xs[2 * h])));
      float sn, cs;
      sincospif(2.0f * uniform23(xs[2 * h + 1]), &sn, &cs);
      r[4 * j + 2 * h] = rad * cs;
      r[4 * j + 2 * h + 1] = rad * sn;
    }
  }
  const float sr = sqrtf(rho);
  float t[15];
#pragma unroll
  for (int k = 0; k < 15; ++k) t[k] = ph.fl_amp[k] * sr * r[k];
#pragma unroll
  for (int p = 0; p < kQ; ++p) {
    float acc = 0.f;
#pragma unroll
    for (int k = 4; k < kQ; ++k)
      if (mode_row(k, p) != 0) acc = fmaf((float)mode_row(k, p), t[k - 4], acc);
    xi[p] = wq(p) * acc;
  }
}

// kNoisePair.  thermal_source_t returns v_p = xi_p / w_p.  The sum over modes
// (mode_row) is taken by the parity of the modes and of the directions: 55
// additions in place of 238 products.
template <class O>
__device__ __forceinline__ void thermal_normals_t(const LbPhys &ph, const uint32_t *node,
                                                  typename O::V r[16]) {
  const long long step = *ph.step;
#pragma unroll
  for (uint32_t j = 0; j < 4; ++j) {
    uint32_t xs[4][O::N];
#pragma unroll
    for (int n = 0; n < O::N; ++n) {
      const U4 c{node[n], (uint32_t)(unsigned long long)step,
                 (uint32_t)((unsigned long long)step >> 32), j | (2u << 8)};
      const U4 x = philox4x32_10(c, (uint32_t)ph.seed, (uint32_t)(ph.seed >> 32));
      xs[0][n] = x.x;
      xs[1][n] = x.y;
      xs[2][n] = x.z;
      xs[3][n] = x.w;
    }
#pragma unroll
    for (int h = 0; h < 2; ++h)
      box_muller_t<O>(uniform23_t<O>(xs[2 * h]), uniform23_t<O>(xs[2 * h + 1]), r[4 * j + 2 * h],
                      r[4 * j + 2 * h + 1]);
  }
}
template <class O>
__device__ __forceinline__ void thermal_source_t(const LbPhys &ph, const typename O::V r[16],
                                                 typename O::V rho, typename O::V v[kQ]) {
  using V = typename O::V;
  float rr[O::N];
  O::unpack(rho, rr);
#pragma unroll
  for (int n = 0; n < O::N; ++n) rr[n] = sqrtf(rr[n]);
  const V sr = O::pack(rr);
  // Products that meet a sum are written as fused operations: paired products
  // (unlike __fmul_rn) are contracted with a sum that follows, and one and two
  // nodes at a time must round alike.
  const auto a = [&](int k) { return O::mul(O::splat(ph.fl_amp[k - 4]), sr); };
  const auto n = [&](int k) { return r[k - 4]; };
  const V two = O::splat(2.0f);
  // directions +-: even part of the modes, plus or minus the odd part
  const auto pair = [&](int p, V even, V odd) {
    v[p] = O::add(even, odd);
    v[p + 1] = O::sub(even, odd);
  };
  const auto axis = [&](int p, V even, int k) {
    const V c = O::mul(O::splat(-2.0f), a(k));
    v[p] = O::fma(c, n(k), even);
    v[p + 1] = O::fma(O::neg(c), n(k), even);
  };
  const V t16 = O::mul(a(16), n(16)), t17 = O::mul(a(17), n(17)), t18 = O::mul(a(18), n(18));
  const V m16 = O::mul(O::splat(-2.0f), t16);
  v[0] = O::fma(O::neg(a(4)), n(4), t16);
  const V a5 = O::fma(a(5), n(5), O::neg(t17)), b5 = O::fma(a(5), n(5), t17);
  const V a6 = O::fma(a(6), n(6), O::neg(t18)), b6 = O::fma(a(6), n(6), t18);
  const V b0 = O::fma(a(4), n(4), t16);
  axis(1, O::fma(two, a5, m16), 10);
  axis(3, O::add(O::sub(a6, a5), m16), 11);
  axis(5, O::sub(m16, O::add(a5, a6)), 12);
  const V t13 = O::mul(a(13), n(13)), t14 = O::mul(a(14), n(14)), t15 = O::mul(a(15), n(15));
  const V xp = O::fma(a(10), n(10), t13), xm = O::fma(a(10), n(10), O::neg(t13));
  const V yp = O::fma(a(11), n(11), t14), ym = O::fma(a(11), n(11), O::neg(t14));
  const V zp = O::fma(a(12), n(12), t15), zm = O::fma(a(12), n(12), O::neg(t15));
  const V bxy = O::add(b0, O::add(b5, b6)), bxz = O::add(b0, O::sub(b5, b6)),
          byz = O::fma(O::splat(-2.0f), b5, b0);
  pair(7, O::fma(a(7), n(7), bxy), O::add(xp, ym));
  pair(9, O::fma(O::neg(a(7)), n(7), bxy), O::sub(xp, ym));
  pair(11, O::fma(a(9), n(9), bxz), O::add(xm, zp));
  pair(13, O::fma(O::neg(a(9)), n(9), bxz), O::sub(xm, zp));
  pair(15, O::fma(a(8), n(8), byz), O::add(yp, zm));
  pair(17, O::fma(O::neg(a(8)), n(8), byz), O::sub(yp, zm));
}

// rho - rho0 and j = sum_p h_p c_p, each a sum in the population order, the
// momentum components as signed sums (no products with c_p).
template <class O>
__device__ __forceinline__ void moments_t(const typename O::V h[kQ], typename O::V &drho,
                                          typename O::V &jx, typename O::V &jy, typename O::V &jz) {
  drho = h[0];
  jx = h[1];
  jy = h[3];
  jz = h[5];
#pragma unroll
  for (int p = 1; p < kQ; ++p) {
    drho = O::add(drho, h[p]);
    if (p != 1 && cx(p) != 0) jx = cx(p) > 0 ? O::add(jx, h[p]) : O::sub(jx, h[p]);
    if (p != 3 && cy(p) != 0) jy = cy(p) > 0 ? O::add(jy, h[p]) : O::sub(jy, h[p]);
    if (p != 5 && cz(p) != 0) jz = cz(p) > 0 ? O::add(jz, h[p]) : O::sub(jz, h[p]);
  }
}

// c_p . u for odd p (the first nonzero component of c_p is +1) as a signed sum.
template <class O>
__device__ __forceinline__ typename O::V cdotu_t(int p, typename O::V ux, typename O::V uy,
                                                 typename O::V uz) {
  typename O::V r = cx(p) != 0 ? ux : (cy(p) != 0 ? uy : uz);
  if (cx(p) != 0 && cy(p) != 0) r = cy(p) > 0 ? O::add(r, uy) : O::sub(r, uy);
  if ((cx(p) != 0 || cy(p) != 0) && cz(p) != 0) r = cz(p) > 0 ? O::add(r, uz) : O::sub(r, uz);
  return r;
}

// Post-collision deviation of every population of one node (or two, Ops2)
// from its pre-collision deviations (Eq. 5, omega = 1/tau, Delta t = 1):
//   h*_p = (1 - omega) h_p + omega heq_p + S_p,
//   heq_p = w_p [ (rho - rho0) + rho (3 c.u + 9/2 (c.u)^2 - 3/2 u.u) ]   (Eq. 6),
//   paper forcing: S_p = 3 w_p c_p . g;
//   Guo forcing:   u = (j + g/2)/rho, S_p = (1 - omega/2) w_p [3 (c - u) + 9 (c.u) c] . g;
//   kForcingNone (g = 0): u = j/rho, S_p = 0;
//   NOISE: plus the thermal source F_p of Eq. 5, of node `node` (kNoiseNode: Ops1
//   only) or from the node's (nodes') fifteen normals (kNoisePair).
// Opposite directions p, opp(p) = p + 1 (odd p) share c.u up to the sign, so
// heq splits into the even part w_p [(rho - rho0) - 3/2 rho u.u + 9/2 rho (c.u)^2]
// and the odd part +-3 w_p rho c.u, computed once per pair.  A node whose
// density is not finite (a population is not) sets *ph.nonfinite.
template <class O, int FORCING, int NOISE = kNoNoise>
__device__ __forceinline__ void collide_t(typename O::V h[kQ], const LbPhys &ph, uint32_t node = 0,
                                          const typename O::V *normals = nullptr) {
  using V = typename O::V;
  static_assert(NOISE != kNoiseNode || O::N == 1, "one node per call");
  V drho, jx, jy, jz;
  moments_t<O>(h, drho, jx, jy, jz);
  const V rho = O::add(O::splat(ph.rho0), drho);
  // one compare and a predicated store per node
  if (!O::finite(rho)) *ph.nonfinite = 1;
  const V inv = O::rcp(rho);
  V ux, uy, uz;
  if (FORCING == LBMD_FORCING_GUO) {
    ux = O::mul(O::fma(O::splat(0.5f), O::splat(ph.g[0]), jx), inv);
    uy = O::mul(O::fma(O::splat(0.5f), O::splat(ph.g[1]), jy), inv);
    uz = O::mul(O::fma(O::splat(0.5f), O::splat(ph.g[2]), jz), inv);
  } else {
    ux = O::mul(jx, inv);
    uy = O::mul(jy, inv);
    uz = O::mul(jz, inv);
  }
  const float om = ph.omega, om1 = 1.0f - om;
  const V vom1 = O::splat(om1);
  const V usq = O::fma(uz, uz, O::fma(uy, uy, O::mul(ux, ux)));
  const V A = O::fma(O::neg(O::mul(O::splat(1.5f), rho)), usq, drho);
  const V r3 = O::mul(O::splat(3.0f), rho), r45 = O::mul(O::splat(4.5f), rho);
  V gu = O::splat(0.f);
  if (FORCING == LBMD_FORCING_GUO)
    gu = O::fma(O::splat(ph.g[2]), uz, O::fma(O::splat(ph.g[1]), uy, O::mul(O::splat(ph.g[0]), ux)));
  const float kguo = fmaf(-0.5f, om, 1.0f);
  // h*_p from the relaxed part, plus the source S_p (c_p . u = cu)
  auto add_source = [&](int p, V cu, V v) -> V {
    const float cg = cx(p) * ph.g[0] + cy(p) * ph.g[1] + cz(p) * ph.g[2];  // one value per kernel
    if (FORCING == LBMD_FORCING_GUO) {
      const V t = O::fma(O::mul(O::splat(9.0f), cu), O::splat(cg),
                         O::mul(O::splat(3.0f), O::sub(O::splat(cg), gu)));
      return O::add(v, O::mul(O::splat(__fmul_rn(kguo, wq(p))), t));
    }
    if (FORCING == LBMD_FORCING_PAPER) return O::add(v, O::splat(__fmul_rn(3.0f * wq(p), cg)));
    return v;
  };
  V xi[kQ];  // F_p, or F_p / w_p
  if constexpr (NOISE == kNoiseNode) thermal_source(ph, node, rho, xi);
  if constexpr (NOISE == kNoisePair) thermal_source_t<O>(ph, normals, rho, xi);
  const auto add_noise = [&](int p) {
    if constexpr (NOISE == kNoiseNode) h[p] = O::add(h[p], xi[p]);
    if constexpr (NOISE == kNoisePair) h[p] = O::fma(O::splat(wq(p)), xi[p], h[p]);
  };
  h[0] = add_source(0, O::splat(0.f), O::fma(O::splat(__fmul_rn(om, wq(0))), A, O::mul(vom1, h[0])));
  add_noise(0);
#pragma unroll
  for (int p = 1; p < kQ; p += 2) {
    const V cu = cdotu_t<O>(p, ux, uy, uz);  // c_opp(p) . u = -cu
    const V even = O::fma(O::mul(r45, cu), cu, A);
    const V ow = O::splat(__fmul_rn(om, wq(p)));
    h[p] = add_source(p, cu, O::fma(ow, O::fma(r3, cu, even), O::mul(vom1, h[p])));
    h[p + 1] = add_source(p + 1, O::neg(cu), O::fma(ow, O::fma(O::neg(r3), cu, even), O::mul(vom1, h[p + 1])));
    add_noise(p);
    add_noise(p + 1);
  }
}

template <int FORCING, int NOISE = kNoNoise>
__device__ __forceinline__ void collide19(float h[kQ], const LbPhys &ph, uint32_t node = 0) {
  float r[16];
  if constexpr (NOISE == kNoisePair) thermal_normals_t<Ops1>(ph, &node, r);
  collide_t<Ops1, FORCING, NOISE>(h, ph, node, r);
}

__device__ __forceinline__ void zero19(float h[kQ]) {
#pragma unroll
  for (int p = 0; p < kQ; ++p) h[p] = 0.f;
}

// Solid nodes are left out, or (LbGeom::fill_solid, except rows that are solid
// as a whole) written as zero, so that the 32-byte sectors they share with fluid
// nodes are written whole: memory completes a sector written in part by a read.
// 256x128x128 with one wall layer, FP32: 99.4-100.7 us a step left out, 94.8-95.0
// filled; boxes that stay in L2 lose by it (48x96x96: 10.6 against 11.0 us).
__device__ __forceinline__ bool solid_is_left_out(const LbGeom &g, int y) {
  return !g.fill_solid || (g.wall.y_walls && (y == 0 || y == g.ny - 1));
}

// Stream and collide node (x, y, z) of one box: pull, Eq. 5 collision, store.
template <int S, int FORCING, typename I, int NOISE = kNoNoise>
__device__ __forceinline__ void stream_collide_node(const LbGeom &g, const LbPhys &ph,
                                                    const typename Store<S>::T *__restrict__ src,
                                                    typename Store<S>::T *__restrict__ dst, int x,
                                                    int y, int z) {
  using St = Store<S>;
  const I self = ((I)z * g.ny + y) * g.nx + x;
  float h[kQ];
  uint32_t bb = 0u;
  // warps with a node beside a wall select their sources by the link mask (the
  // others' loads wait for nothing)
  if (__any_sync(__activemask(), beside_wall(g, x, y))) {
    if (beside_wall(g, x, y)) bb = __ldg(&g.lmask[self]);
    if ((bb & 1u) && solid_is_left_out(g, y)) return;
    pull19_mask<S, I>(g, src, x, y, z, bb, h);
    if (bb & 1u) zero19(h);
  } else {
    pull19_mask<S, I>(g, src, x, y, z, 0u, h);  // constant mask: no selects
  }
  collide19<FORCING, NOISE>(h, ph, (uint32_t)self);
  if (bb & 1u) zero19(h);
  const I st = pop_stride<S, I>((I)g.Vp);
  const I at = pop_base<S, I>(((I)z * g.ny + y) * row_pitch<S>(g) + x);
#pragma unroll
  for (int p = 0; p < kQ; ++p) St::store(dst + (I)p * st + at, h[p]);
}


// Nodes (x, y, z) and (x, y, z + 1) of one box (z + 1 < nz), with all 38
// loads issued before either collision.
template <int S, int FORCING>
__device__ __forceinline__ void stream_collide_node2(const LbGeom &g, const LbPhys &ph,
                                                     const typename Store<S>::T *__restrict__ src,
                                                     typename Store<S>::T *__restrict__ dst, int x,
                                                     int y, int z) {
  using St = Store<S>;
  const int self_a = (z * g.ny + y) * g.nx + x, self_b = self_a + g.nx * g.ny;
  float ha[kQ], hb[kQ];
  uint32_t ma = 0u, mb = 0u;
  if (beside_wall(g, x, y)) {
    ma = __ldg(&g.lmask[self_a]);
    mb = __ldg(&g.lmask[self_b]);
  }
  pull19_mask<S, int>(g, src, x, y, z, 0u, ha);  // constant masks: no selects
  pull19_mask<S, int>(g, src, x, y, z + 1, 0u, hb);
  const int own_a = (z * g.ny + y) * row_pitch<S>(g) + x, own_b = own_a + row_pitch<S>(g) * g.ny;
  if (ma) bounce19<S, int>(g, src, own_a, ma, ha);
  if (mb) bounce19<S, int>(g, src, own_b, mb, hb);
  const int st = pop_stride<S, int>((int)g.Vp);
  if (!(ma & 1u)) {  // a solid node is pulled but not written
    collide19<FORCING>(ha, ph);
#pragma unroll
    for (int p = 0; p < kQ; ++p) St::store(dst + p * st + pop_base<S, int>(own_a), ha[p]);
  }
  if (!(mb & 1u)) {
    collide19<FORCING>(hb, ph);
#pragma unroll
    for (int p = 0; p < kQ; ++p) St::store(dst + p * st + pop_base<S, int>(own_b), hb[p]);
  }
}

// 16-bit storage, two x-adjacent nodes (2 xw, 2 xw + 1) of one box per
// call: their deviations of one population share a 32-bit word (rows are held
// at an even length, so a pair never straddles a row; the second node of an odd
// row's last pair is padding).  Every population is one 32-bit load for
// c_x = 0 and two for c_x = +-1 (the neighbouring word supplies the shifted
// half; one byte permute assembles the pair), one 32-bit store, and the
// collision runs once for both nodes on float2 with the paired FP32
// instructions -- the same bits as stream_collide_node for either node.
// Word offsets are 32-bit (19 Vp < 2^31).
template <typename T2> struct Pair16;
template <> struct Pair16<__half2> {
  static __device__ __forceinline__ float2 unpack(uint32_t w) {
    return __half22float2(*reinterpret_cast<const __half2 *>(&w));
  }
  static __device__ __forceinline__ uint32_t pack(float2 v) {
    const __half2 h = __float22half2_rn(v);
    return *reinterpret_cast<const uint32_t *>(&h);
  }
};
template <> struct Pair16<__nv_bfloat162> {
  static __device__ __forceinline__ float2 unpack(uint32_t w) {
    return __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&w));
  }
  static __device__ __forceinline__ uint32_t pack(float2 v) {
    const __nv_bfloat162 h = __float22bfloat162_rn(v);
    return *reinterpret_cast<const uint32_t *>(&h);
  }
};

// The populations that bounce back (bits p of bb) from the pair's own words `own`:
// of opp(p), or of p with SWAPPED (in place).  All words are read, six at a time
// in flight, and those that bounce are taken: a branch for each direction, which
// the compiler makes of the plain form, waits for one read after another
// (256x128x128 with a wall, a step: FP16 59.6 -> 57.1 us, BF16 63 -> 57.0; 32^3 with
// a wall 3.4 -> 3.0, BF16 4.5 -> 3.0).  In place the buffer is written by the same kernel: no read-only path.
template <typename T2, bool SWAPPED>
__device__ __forceinline__ void pair_bounce(const uint32_t *own, uint2 bb, float2 h[kQ]) {
  constexpr int kW = kBlockNodes / 2, kB = 6;
#pragma unroll
  for (int p0 = 1; p0 < kQ; p0 += kB) {
    uint32_t r[kB];
#pragma unroll
    for (int k = 0; k < kB; ++k) {
      const uint32_t *q = own + (SWAPPED ? p0 + k : opp(p0 + k)) * kW;
      if (SWAPPED)
        asm volatile("ld.global.u32 %0, [%1];" : "=r"(r[k]) : "l"(q));
      else
        asm volatile("ld.global.nc.u32 %0, [%1];" : "=r"(r[k]) : "l"(q));
    }
#pragma unroll
    for (int k = 0; k < kB; ++k) {
      const int p = p0 + k;
      const float2 v = Pair16<T2>::unpack(r[k]);
      h[p].x = ((bb.x >> p) & 1u) ? v.x : h[p].x;
      h[p].y = ((bb.y >> p) & 1u) ? v.y : h[p].y;
    }
  }
}

// pair_pull: the pre-collision deviations h of both nodes (zero for a solid one
// and for padding); returns their link masks.
template <typename T2>
__device__ __forceinline__ uint2 pair_pull(const LbGeom &g, const uint32_t *__restrict__ src, int xw,
                                           int y, int z, float2 h[kQ]) {
  using P = Pair16<T2>;
  const int wpr = g.pitch >> 1;  // words per row
  const bool odd = g.nx & 1, lone = odd && xw == wpr - 1;
  // a word w of the node pairs' row-major order, population p: words of
  // pop_base's blocks (32 words a population)
  constexpr int kW = kBlockNodes / 2;
  const auto word = [](const uint32_t *b, int w) { return b + (w + (w >> 5) * ((kQ - 1) * kW)); };
  const int ny = g.ny;
  const int self = (z * ny + y) * wpr + xw;
  const int ym = wrap_m1(y, ny), yp = wrap_p1(y, ny);
  const int zm = wrap_m1(z, g.nz), zp = wrap_p1(z, g.nz);
  const int xl = xw == 0 ? wpr - 1 : xw - 1, xr = xw == wpr - 1 ? 0 : xw + 1;
  // link masks of the two nodes (bit 0: solid; bit p: the pull source is solid)
  uint2 bb = make_uint2(0u, 0u);
  if (beside_wall<2>(g, 2 * xw, y)) {
    const uint32_t *m = g.lmask + ((z * ny + y) * g.nx + 2 * xw);
    bb.x = __ldg(m);
    if (!lone) bb.y = __ldg(m + 1);
  }
#pragma unroll
  for (int p = 0; p < kQ; ++p) {
    // source row of x - c_p; the pair's sources are x - c_x, x - c_x + 1
    const int sy = cy(p) == 1 ? ym : (cy(p) == -1 ? yp : y);
    const int sz = cz(p) == 1 ? zm : (cz(p) == -1 ? zp : z);
    const int row = (sz * ny + sy) * wpr;
    const uint32_t w0 = __ldg(word(src, row + xw) + p * kW);
    uint32_t w = w0;
    // (x - 1, x): node nx - 1 of an odd row is the first of its word
    if (cx(p) == 1) w = __byte_perm(__ldg(word(src, row + xl) + p * kW), w0, odd && xw == 0 ? 0x5410 : 0x5432);
    // (x + 1, x + 2): behind the last node of an odd row comes the first one
    if (cx(p) == -1) w = __byte_perm(w0, __ldg(word(src, row + xr) + p * kW), lone ? 0x5454 : 0x5432);
    h[p] = P::unpack(w);
  }
  if (lone)  // padding: harmless inputs
#pragma unroll
    for (int p = 0; p < kQ; ++p) h[p].y = 0.f;
  if (bb.x | bb.y) {
    // halfway bounce-back: a population whose source is solid comes back as
    // the node's own post-collision opposite population
    pair_bounce<T2, false>(word(src, self), bb, h);
    // a solid node of the pair: harmless inputs, and zero written back
    if (bb.x & 1u)
#pragma unroll
      for (int p = 0; p < kQ; ++p) h[p].x = 0.f;
    if (bb.y & 1u)
#pragma unroll
      for (int p = 0; p < kQ; ++p) h[p].y = 0.f;
  }
  return bb;
}

template <typename T2, int FORCING>
__device__ __forceinline__ void pair_node(const LbGeom &g, const LbPhys &ph,
                                          const uint32_t *__restrict__ src,
                                          uint32_t *__restrict__ dst, int xw, int y, int z) {
  using P = Pair16<T2>;
  constexpr int kW = kBlockNodes / 2;
  float2 h[kQ];
  const uint2 bb = pair_pull<T2>(g, src, xw, y, z, h);
  const int self = (z * g.ny + y) * (g.pitch >> 1) + xw;
  collide_t<Ops2, FORCING>(h, ph);
  if ((bb.x | bb.y) & 1u) {
    if (bb.x & 1u)
#pragma unroll
      for (int p = 0; p < kQ; ++p) h[p].x = 0.f;
    if (bb.y & 1u)
#pragma unroll
      for (int p = 0; p < kQ; ++p) h[p].y = 0.f;
  }
  uint32_t *out = dst + (self + (self >> 5) * ((kQ - 1) * kW));
#pragma unroll
  for (int p = 0; p < kQ; ++p) out[p * kW] = P::pack(h[p]);
}

}  // namespace lbmd
