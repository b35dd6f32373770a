// lb_fluct.cu -- the stream-collide with the thermal source F_p of Eq. 5
// (fluctuating LB), in its own translation unit: the same node update as
// k_stream_collide (pull) or k_aa_stream_collide (in place) plus fifteen
// Philox normals per node.
#include <cmath>

#include "lb_aa.cuh"

namespace lbmd {

// Two nodes per thread, on consecutive z-planes, for the paired FP32
// instructions: the noise is bound by instructions (~1300 per node with the
// library's logarithm, sine and root one node at a time, 780 now; two fifths
// of the FMA pipe's time are Philox products).  The normals are drawn before
// the 38 loads are issued, so that both fit 96 registers: five blocks of 128
// threads.  128^3, FP32: 92 us a step before, 71 now; 74 with six blocks (80
// registers, spills), 77 with the loads first and 16 warps per SM.  An odd last
// plane is taken alone.  EARLY, for boxes of up to 2^15 nodes, where latency
// counts: the loads first, the normals while they are under way (32^3, FP32 4.4 ->
// 4.25 us a step, with a wall 5.7 -> 5.15; 40^3 is slower by it, 6.6 -> 6.7).
constexpr int kFluctRows = 4;

// bounce19 with all words read, six in flight, and those that bounce taken (a
// branch for each direction waits for one read after another).
template <int S, typename I>
__device__ __forceinline__ void bounce_six(const LbGeom &g, const typename Store<S>::T *__restrict__ src,
                                           I self, uint32_t bb, float h[kQ]) {
  const I st = pop_stride<S, I>((I)g.Vp);
  const typename Store<S>::T *own = src + pop_base<S, I>(self);
#pragma unroll
  for (int p0 = 1; p0 < kQ; p0 += 6) {
    float r[6];
#pragma unroll
    for (int k = 0; k < 6; ++k) r[k] = Store<S>::load(own + (I)opp(p0 + k) * st);
#pragma unroll
    for (int k = 0; k < 6; ++k) asm volatile("" : "+f"(r[k]));  // read before any is chosen
#pragma unroll
    for (int k = 0; k < 6; ++k) h[p0 + k] = ((bb >> (p0 + k)) & 1u) ? r[k] : h[p0 + k];
  }
}

template <int S, int FORCING, typename I, bool EARLY>
__global__ void __launch_bounds__(32 * kFluctRows, EARLY ? 2 : 5)
    k_stream_collide_fluct(LbGeom g, LbPhys ph, const typename Store<S>::T *__restrict__ src,
                           typename Store<S>::T *__restrict__ dst) {
  using St = Store<S>;
  const int x = blockIdx.x * 32 + threadIdx.x;
  const int y = blockIdx.y * kFluctRows + threadIdx.y;
  const int za = 2 * blockIdx.z, zb = min(za + 1, g.nz - 1);
  if (x >= g.nx || y >= g.ny) return;
  const I na = ((I)za * g.ny + y) * g.nx + x, nb = ((I)zb * g.ny + y) * g.nx + x;
  uint32_t ma = 0u, mb = 0u;
  if (beside_wall(g, x, y)) {
    ma = __ldg(&g.lmask[na]);
    mb = __ldg(&g.lmask[nb]);
  }
  if (ma & mb & 1u) return;
  const uint32_t node[2] = {(uint32_t)na, (uint32_t)nb};
  float2 r[16];
  if (!EARLY) thermal_normals_t<Ops2>(ph, node, r);
  float ha[kQ], hb[kQ];
  pull19_mask<S, I>(g, src, x, y, za, 0u, ha);
  pull19_mask<S, I>(g, src, x, y, zb, 0u, hb);
  if (EARLY) thermal_normals_t<Ops2>(ph, node, r);
  const I oa = ((I)za * g.ny + y) * row_pitch<S>(g) + x, ob = ((I)zb * g.ny + y) * row_pitch<S>(g) + x;
  if (EARLY || S == LBMD_STORE_F32) {
    if (ma | mb) {
      bounce_six<S, I>(g, src, oa, ma, ha);
      bounce_six<S, I>(g, src, ob, mb, hb);
    }
  } else {  // 16-bit words at 96 registers: six in flight spill
    if (ma) bounce19<S, I>(g, src, oa, ma, ha);
    if (mb) bounce19<S, I>(g, src, ob, mb, hb);
  }
  if (ma & 1u) zero19(ha);  // harmless inputs: not written
  if (mb & 1u) zero19(hb);
  float2 h[kQ];
#pragma unroll
  for (int p = 0; p < kQ; ++p) h[p] = make_float2(ha[p], hb[p]);
  collide_t<Ops2, FORCING, true>(h, ph, r);
  const I st = pop_stride<S, I>((I)g.Vp);
  if (!(ma & 1u)) {
    typename St::T *out = dst + pop_base<S, I>(oa);
#pragma unroll
    for (int p = 0; p < kQ; ++p) St::store(out + (I)p * st, h[p].x);
  }
  if (zb != za && !(mb & 1u)) {
    typename St::T *out = dst + pop_base<S, I>(ob);
#pragma unroll
    for (int p = 0; p < kQ; ++p) St::store(out + (I)p * st, h[p].y);
  }
}

template <int S, typename I, bool EARLY>
static cudaError_t fluct_launch(const LbGeom &g, const LbPhys &ph, const void *src, void *dst,
                                cudaStream_t s) {
  using T = typename Store<S>::T;
  dim3 block(32, kFluctRows);
  dim3 grid(g.ntx, (g.ny + kFluctRows - 1) / kFluctRows, (g.nz + 1) / 2);
  const T *a = (const T *)src;
  T *b = (T *)dst;
  if (ph.g[0] == 0.f && ph.g[1] == 0.f && ph.g[2] == 0.f)
    k_stream_collide_fluct<S, kForcingNone, I, EARLY><<<grid, block, 0, s>>>(g, ph, a, b);
  else if (ph.forcing == LBMD_FORCING_GUO)
    k_stream_collide_fluct<S, LBMD_FORCING_GUO, I, EARLY><<<grid, block, 0, s>>>(g, ph, a, b);
  else
    k_stream_collide_fluct<S, LBMD_FORCING_PAPER, I, EARLY><<<grid, block, 0, s>>>(g, ph, a, b);
  return cudaGetLastError();
}

template <int S>
static cudaError_t fluct_launch(const LbGeom &g, const LbPhys &ph, const void *src, void *dst,
                                cudaStream_t s) {
  if ((long long)g.nx * g.ny * g.nz <= 1 << 15) return fluct_launch<S, int, true>(g, ph, src, dst, s);
  if ((long long)kQ * g.Vp < 0x7fffffffLL) return fluct_launch<S, int, false>(g, ph, src, dst, s);
  return fluct_launch<S, size_t, false>(g, ph, src, dst, s);
}

cudaError_t launch_lb_stream_collide_fluct(int storage, const LbGeom &g, const LbPhys &ph,
                                           const void *src, void *dst, cudaStream_t s) {
  switch (storage) {
    case LBMD_STORE_F32: return fluct_launch<LBMD_STORE_F32>(g, ph, src, dst, s);
    case LBMD_STORE_F16: return fluct_launch<LBMD_STORE_F16>(g, ph, src, dst, s);
    case LBMD_STORE_BF16: return fluct_launch<LBMD_STORE_BF16>(g, ph, src, dst, s);
  }
  return cudaErrorInvalidValue;
}

cudaError_t launch_lb_aa_fluct(int storage, const LbGeom &g, const LbPhys &ph, void *buf,
                               int odd, cudaStream_t s) {
  return aa_launch_storage<true>(storage, g, ph, buf, odd, nullptr, s);
}

void fluct_amplitudes(double kT, double tau, float amp[15]) {
  const double g1 = 1.0 - 1.0 / tau;
  for (int k = 4; k < kQ; ++k) {
    double b = 0.0;  // b_k = sum_p w_p e_kp^2
    for (int p = 0; p < kQ; ++p) b += (double)wq(p) * mode_row(k, p) * mode_row(k, p);
    amp[k - 4] = (float)std::sqrt(3.0 * kT * (1.0 - g1 * g1) / b);
  }
}

__global__ void k_bump_step(DevStatus *status) { status->step += 1; }

cudaError_t launch_bump_step(DevStatus *status, cudaStream_t s) {
  k_bump_step<<<1, 1, 0, s>>>(status);
  return cudaGetLastError();
}

}  // namespace lbmd
