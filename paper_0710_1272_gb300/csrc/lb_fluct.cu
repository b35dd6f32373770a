// lb_fluct.cu -- the stream-collide with the thermal source F_p of Eq. 5
// (fluctuating LB), in its own translation unit: the same node update as
// k_stream_collide (pull) or k_aa_stream_collide (in place) plus fifteen
// Philox normals per node.
#include <algorithm>
#include <cmath>

#include "lb_aa.cuh"

namespace lbmd {

// One node per thread (kNoiseNode): 16-bit storage, and boxes with a chain.
// Bound by the noise's instructions: 128^3 FP16 92 us a step, in place 101.
template <int S, int FORCING, typename I>
__global__ void __launch_bounds__(32 * kRowsPerBlock)
    k_stream_collide_fluct_node(LbGeom g, LbPhys ph, const typename Store<S>::T *__restrict__ src,
                                typename Store<S>::T *__restrict__ dst) {
  const int x = blockIdx.x * 32 + threadIdx.x;
  const int y = blockIdx.y * kRowsPerBlock + threadIdx.y;
  const int z = blockIdx.z;
  if (x >= g.nx || y >= g.ny) return;
  stream_collide_node<S, FORCING, I, kNoiseNode>(g, ph, src, dst, x, y, z);
}

// FP32 solvent (kNoisePair): two nodes per thread, on consecutive z-planes, for
// the paired FP32 instructions: the noise is bound by instructions (~1300 per
// node with the library's logarithm, sine and root one node at a time, 780 now;
// two fifths of the FMA pipe's time are Philox products).  The normals are drawn
// before the 38 loads are issued, so that both fit 96 registers: five blocks of
// 128 threads.  128^3: 92 us a step before, 68 now; 74 with six blocks (80
// registers, spills), 77 with the loads first and 16 warps per SM.  An odd last
// plane is taken alone.  EARLY, for boxes of up to 2^15 nodes, where latency
// counts: the loads first, the normals while they are under way (32^3 4.4 ->
// 4.25 us a step, with a wall 5.7 -> 5.15; 40^3 is slower by it, 6.6 -> 6.7).
constexpr int kFluctRows = 4;

// bounce19 with all words read, six in flight, and those that bounce taken (a
// branch for each direction waits for one read after another).
template <typename I>
__device__ __forceinline__ void bounce_six(const LbGeom &g, const float *__restrict__ src, I self, uint32_t bb,
                                           float h[kQ]) {
  const I st = (I)g.Vp;
  const float *own = src + self;
#pragma unroll
  for (int p0 = 1; p0 < kQ; p0 += 6) {
    float r[6];
#pragma unroll
    for (int k = 0; k < 6; ++k) r[k] = __ldg(own + (I)opp(p0 + k) * st);
#pragma unroll
    for (int k = 0; k < 6; ++k) asm volatile("" : "+f"(r[k]));  // read before any is chosen
#pragma unroll
    for (int k = 0; k < 6; ++k) h[p0 + k] = ((bb >> (p0 + k)) & 1u) ? r[k] : h[p0 + k];
  }
}

template <int FORCING, typename I, bool EARLY>
__global__ void __launch_bounds__(32 * kFluctRows, EARLY ? 2 : 5)
    k_stream_collide_fluct(LbGeom g, LbPhys ph, int y0, const float *__restrict__ src,
                           float *__restrict__ dst) {
  const int x = blockIdx.x * 32 + threadIdx.x;
  const int y = y0 + blockIdx.y * kFluctRows + threadIdx.y;
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
  pull19_mask<LBMD_STORE_F32, I>(g, src, x, y, za, 0u, ha);
  pull19_mask<LBMD_STORE_F32, I>(g, src, x, y, zb, 0u, hb);
  if (EARLY) thermal_normals_t<Ops2>(ph, node, r);
  if (ma | mb) {
    bounce_six<I>(g, src, na, ma, ha);
    bounce_six<I>(g, src, nb, mb, hb);
  }
  if (ma & 1u) zero19(ha);  // harmless inputs: not written
  if (mb & 1u) zero19(hb);
  float2 h[kQ];
#pragma unroll
  for (int p = 0; p < kQ; ++p) h[p] = make_float2(ha[p], hb[p]);
  collide_t<Ops2, FORCING, kNoisePair>(h, ph, 0, r);
  const I st = (I)g.Vp;
  if (!(ma & 1u))
#pragma unroll
    for (int p = 0; p < kQ; ++p) dst[na + (I)p * st] = h[p].x;
  if (zb != za && !(mb & 1u))
#pragma unroll
    for (int p = 0; p < kQ; ++p) dst[nb + (I)p * st] = h[p].y;
}

template <typename I, bool EARLY>
static cudaError_t fluct_launch_pair(const LbGeom &g, const LbPhys &ph, const void *src, void *dst,
                                     cudaStream_t s) {
  dim3 block(32, kFluctRows);
  const float *a = (const float *)src;
  float *b = (float *)dst;
  // the grid's 65535 rows of blocks are half as many nodes as the other
  // kernels': boxes of ny > 262140 take two launches
  for (int y0 = 0; y0 < g.ny; y0 += 65535 * kFluctRows) {
    dim3 grid(g.ntx, std::min((g.ny - y0 + kFluctRows - 1) / kFluctRows, 65535), (g.nz + 1) / 2);
    if (ph.g[0] == 0.f && ph.g[1] == 0.f && ph.g[2] == 0.f)
      k_stream_collide_fluct<kForcingNone, I, EARLY><<<grid, block, 0, s>>>(g, ph, y0, a, b);
    else if (ph.forcing == LBMD_FORCING_GUO)
      k_stream_collide_fluct<LBMD_FORCING_GUO, I, EARLY><<<grid, block, 0, s>>>(g, ph, y0, a, b);
    else
      k_stream_collide_fluct<LBMD_FORCING_PAPER, I, EARLY><<<grid, block, 0, s>>>(g, ph, y0, a, b);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

template <int S, typename I>
static cudaError_t fluct_launch_node(const LbGeom &g, const LbPhys &ph, const void *src, void *dst,
                                     cudaStream_t s) {
  using T = typename Store<S>::T;
  dim3 block(32, kRowsPerBlock);
  dim3 grid(g.ntx, (g.ny + kRowsPerBlock - 1) / kRowsPerBlock, g.nz);
  const T *a = (const T *)src;
  T *b = (T *)dst;
  if (ph.g[0] == 0.f && ph.g[1] == 0.f && ph.g[2] == 0.f)
    k_stream_collide_fluct_node<S, kForcingNone, I><<<grid, block, 0, s>>>(g, ph, a, b);
  else if (ph.forcing == LBMD_FORCING_GUO)
    k_stream_collide_fluct_node<S, LBMD_FORCING_GUO, I><<<grid, block, 0, s>>>(g, ph, a, b);
  else
    k_stream_collide_fluct_node<S, LBMD_FORCING_PAPER, I><<<grid, block, 0, s>>>(g, ph, a, b);
  return cudaGetLastError();
}
template <int S>
static cudaError_t fluct_launch_node(const LbGeom &g, const LbPhys &ph, const void *src, void *dst,
                                     cudaStream_t s) {
  if ((long long)kQ * g.Vp < 0x7fffffffLL) return fluct_launch_node<S, int>(g, ph, src, dst, s);
  return fluct_launch_node<S, size_t>(g, ph, src, dst, s);
}

cudaError_t launch_lb_stream_collide_fluct(int storage, const LbGeom &g, const LbPhys &ph,
                                           const void *src, void *dst, bool chain, cudaStream_t s) {
  if (storage == LBMD_STORE_F32 && !chain) {
    if ((long long)g.nx * g.ny * g.nz <= 1 << 15) return fluct_launch_pair<int, true>(g, ph, src, dst, s);
    if ((long long)kQ * g.Vp < 0x7fffffffLL) return fluct_launch_pair<int, false>(g, ph, src, dst, s);
    return fluct_launch_pair<size_t, false>(g, ph, src, dst, s);
  }
  switch (storage) {
    case LBMD_STORE_F32: return fluct_launch_node<LBMD_STORE_F32>(g, ph, src, dst, s);
    case LBMD_STORE_F16: return fluct_launch_node<LBMD_STORE_F16>(g, ph, src, dst, s);
    case LBMD_STORE_BF16: return fluct_launch_node<LBMD_STORE_BF16>(g, ph, src, dst, s);
  }
  return cudaErrorInvalidValue;
}

cudaError_t launch_lb_aa_fluct(int storage, const LbGeom &g, const LbPhys &ph, void *buf,
                               int odd, bool chain, cudaStream_t s) {
  if (storage == LBMD_STORE_F32 && !chain)
    return aa_launch_f32<kNoisePair>(g, ph, buf, odd, nullptr, s);
  return aa_launch_storage<kNoiseNode>(storage, g, ph, buf, odd, nullptr, s);
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
