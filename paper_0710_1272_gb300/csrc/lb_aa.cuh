// lb_aa.cuh -- in-place (AA-pattern) streaming of the D3Q19 populations
// (Bailey, Myre, Walsh, Lilja and Saar, ICPP 2009): one population buffer
// instead of two, the same Eq. 5 update and the same bytes moved per node.
//
// Two kinds of step alternate, and each reads and writes the same 19 slots
// per node, so every update is race-free in place:
//   even step (buffer kPopAALocal -> kPopAASwap): node x reads its own
//     h_p(x) at [p][x], collides, and writes h*_p(x) to [opp(p)][x];
//   odd step (buffer kPopAASwap -> kPopAALocal): node x pulls
//       h_p(x) = [opp(p)][x - c_p]  (h*_p(x - c_p), streamed), or
//                [p][x]             (h*_opp(p)(x), bounced back) if x - c_p is solid,
//     collides, and pushes h*_p(x) to
//       [p][x + c_p]                (the next even step's h_p(x + c_p)), or
//       [opp(p)][x]                 (its h_opp(p)(x): halfway bounce-back) if x + c_p is solid.
// Re-indexed with q = opp(p), the odd step's write set at x is
// {[opp(q)][x - c_q] : x - c_q fluid} u {[q][x] : x - c_q solid}, its read set;
// a slot belongs to one fluid node only, and no node reads a slot of a solid
// node.  The bounce-back of Eq. 5's pull form is thus reproduced exactly.
//
// The buffer is read and written by the same kernel, so it is accessed
// through a plain (non-restrict, non-const) pointer: no load may take the
// read-only data path.
#pragma once

#include "lb_collide.cuh"

namespace lbmd {

template <int S, int FORCING, typename I, bool ODD, int NOISE>
__device__ __forceinline__ void aa_node(const LbGeom &g, const LbPhys &ph,
                                        typename Store<S>::T *buf, int x, int y, int z,
                                        uint32_t bb) {
  using St = Store<S>;
  const int nx = g.nx, ny = g.ny;
  const int pitch = row_pitch<S>(g);
  const I node = ((I)z * ny + y) * nx + x, self = ((I)z * ny + y) * pitch + x;
  const I st = pop_stride<S, I>((I)g.Vp);
  if (bb & 1u) return;  // solid node
  float h[kQ];
  if (!ODD) {
#pragma unroll
    for (int p = 0; p < kQ; ++p) h[p] = St::load_plain(buf + (I)p * st + pop_base<S, I>(self));
    collide19<FORCING, NOISE>(h, ph, (uint32_t)node);
    // The store addresses are the load addresses permuted; hiding the base
    // behind an empty asm makes the compiler recompute them after the
    // collision instead of keeping 19 of them live across it (which spills).
    typename Store<S>::T *out = buf + pop_base<S, I>(self);
    asm volatile("" : "+l"(out));
#pragma unroll
    for (int p = 0; p < kQ; ++p) St::store(out + (I)opp(p) * st, h[p]);
    return;
  }
  const int xm = wrap_m1(x, nx), xp = wrap_p1(x, nx);
  const int ym = wrap_m1(y, ny), yp = wrap_p1(y, ny);
  const int zm = wrap_m1(z, g.nz), zp = wrap_p1(z, g.nz);
#pragma unroll
  for (int p = 0; p < kQ; ++p) {
    // source node x - c_p
    const int sx = cx(p) == 1 ? xm : (cx(p) == -1 ? xp : x);
    const int sy = cy(p) == 1 ? ym : (cy(p) == -1 ? yp : y);
    const int sz = cz(p) == 1 ? zm : (cz(p) == -1 ? zp : z);
    const I sidx = (I)opp(p) * st + pop_base<S, I>(((I)sz * ny + sy) * pitch + sx);
    const I bidx = (I)p * st + pop_base<S, I>(self);
    h[p] = St::load_plain(buf + (((bb >> p) & 1u) ? bidx : sidx));
  }
  collide19<FORCING, NOISE>(h, ph, (uint32_t)node);
  // As in the even step: the store offsets equal the load offsets of the
  // opposite directions, so the coordinates are hidden behind an empty asm
  // and the offsets recomputed rather than kept live across the collision.
  typename Store<S>::T *out = buf;
  int ox = x, oy = y, oz = z;
  asm volatile("" : "+l"(out), "+r"(ox), "+r"(oy), "+r"(oz));
  const int oxm = wrap_m1(ox, nx), oxp = wrap_p1(ox, nx);
  const int oym = wrap_m1(oy, ny), oyp = wrap_p1(oy, ny);
  const int ozm = wrap_m1(oz, g.nz), ozp = wrap_p1(oz, g.nz);
  const I oself = ((I)oz * ny + oy) * pitch + ox;
#pragma unroll
  for (int p = 0; p < kQ; ++p) {
    // destination node x + c_p; bit opp(p) of the mask: x + c_p is solid
    const int tx = cx(p) == 1 ? oxp : (cx(p) == -1 ? oxm : ox);
    const int ty = cy(p) == 1 ? oyp : (cy(p) == -1 ? oym : oy);
    const int tz = cz(p) == 1 ? ozp : (cz(p) == -1 ? ozm : oz);
    const I didx = (I)p * st + pop_base<S, I>(((I)tz * ny + ty) * pitch + tx);
    const I bidx = (I)opp(p) * st + pop_base<S, I>(oself);
    St::store(out + (((bb >> opp(p)) & 1u) ? bidx : didx), h[p]);
  }
}

// One thread per node, a warp per 32 consecutive x of a row, as the pull
// kernel; without the thermal source six 256-thread blocks per SM for the
// even step and five for the odd step (whose shifted stores need more
// registers: at six it spills, and runs 1.7 % slower on a 256^3 solvent).
template <int S, int FORCING, typename I, bool ODD, int NOISE>
__global__ void __launch_bounds__(32 * kRowsPerBlock, NOISE ? 1 : (ODD ? 5 : 6))
    k_aa_stream_collide(LbGeom g, LbPhys ph, typename Store<S>::T *buf, DevStatus *bump) {
  const int x = blockIdx.x * 32 + threadIdx.x;
  const int y = blockIdx.y * kRowsPerBlock + threadIdx.y;
  const int z = blockIdx.z;
  if (bump != nullptr && x == 0 && y == 0 && z == 0) bump->step += 1;
  if (x >= g.nx || y >= g.ny) return;
  uint32_t bb = 0u;  // link mask; zero away from solid nodes
  if (beside_wall(g, x, y)) bb = __ldg(&g.lmask[((size_t)z * g.ny + y) * g.nx + x]);
  aa_node<S, FORCING, I, ODD, NOISE>(g, ph, buf, x, y, z, bb);
}

// 16-bit storage: the pair of x-adjacent nodes (2 xw, 2 xw + 1) whose deviations
// share a word (pair_node), the same slots and the same bits as aa_node for
// either.  The even step reads and writes whole words.  The odd step reads as
// pair_pull does and pushes whole words for c_x = 0, halves for c_x = +-1 (the
// other half of such a word is another thread's); what it reads of a solid
// node is not used.  Bound by instructions like the pull kernel, of which two
// nodes need not many more than one.  us a step, one node per thread / even step
// by pairs / both: 256x128x128 FP16 71.9 / - / 59.1, with a wall 76.7 / 71.9 /
// 64.7, 192x96x96 with a wall 29.5 / 27.6 / 24.9, 256^3 280 / - / 227.  In the odd step a warp with a wall takes the halves'
// way for most directions, so where one warp in two or three has one, or a box
// is short of warps, the odd step stays with one node per thread: 160x96x96 with
// a wall 24.6 / 24.2 / 24.8, 96x64x64 8.5 / 8.5 / 9.8, 48x96x96 without 10.8 /
// 10.1 / 8.9, 64^3 5.8 / 5.5 / 5.3, 32^3 2.31 / 2.33 / 2.84.
template <typename T2, int S, int FORCING, bool ODD>
__device__ __forceinline__ void aa_pair(const LbGeom &g, const LbPhys &ph, typename Store<S>::T *buf,
                                        int xw, int y, int z) {
  using P = Pair16<T2>;
  using St = Store<S>;
  constexpr int kW = kBlockNodes / 2;
  const int wpr = g.pitch >> 1, nx = g.nx, ny = g.ny;
  const bool odd = nx & 1, lone = odd && xw == wpr - 1;  // lone: the second node is padding
  const int self = (z * ny + y) * wpr + xw;
  uint2 bb = make_uint2(0u, 0u);
  if (beside_wall<2>(g, 2 * xw, y)) {
    const uint32_t *m = g.lmask + ((z * ny + y) * nx + 2 * xw);
    bb.x = __ldg(m);
    if (!lone) bb.y = __ldg(m + 1);
  }
  const auto word = [](int w) { return w + (w >> 5) * ((kQ - 1) * kW); };
  uint32_t *words = reinterpret_cast<uint32_t *>(buf);
  float2 h[kQ];
  const int ym = wrap_m1(y, ny), yp = wrap_p1(y, ny);
  const int zm = wrap_m1(z, g.nz), zp = wrap_p1(z, g.nz);
  if (!ODD) {
#pragma unroll
    for (int p = 0; p < kQ; ++p) h[p] = P::unpack(words[word(self) + p * kW]);
  } else {
    const int xl = xw == 0 ? wpr - 1 : xw - 1, xr = xw == wpr - 1 ? 0 : xw + 1;
#pragma unroll
    for (int p = 0; p < kQ; ++p) {
      const int sy = cy(p) == 1 ? ym : (cy(p) == -1 ? yp : y);
      const int sz = cz(p) == 1 ? zm : (cz(p) == -1 ? zp : z);
      const int row = (sz * ny + sy) * wpr;
      const uint32_t w0 = words[word(row + xw) + opp(p) * kW];
      uint32_t w = w0;
      if (cx(p) == 1) w = __byte_perm(words[word(row + xl) + opp(p) * kW], w0, odd && xw == 0 ? 0x5410 : 0x5432);
      if (cx(p) == -1) w = __byte_perm(w0, words[word(row + xr) + opp(p) * kW], lone ? 0x5454 : 0x5432);
      h[p] = P::unpack(w);
    }
    if (bb.x | bb.y) pair_bounce<T2, true>(words + word(self), bb, h);
  }
  const bool skip_a = bb.x & 1u, skip_b = (bb.y & 1u) || lone;  // solid, or padding
  if (skip_a)
#pragma unroll
    for (int p = 0; p < kQ; ++p) h[p].x = 0.f;
  if (skip_b)
#pragma unroll
    for (int p = 0; p < kQ; ++p) h[p].y = 0.f;
  collide_t<Ops2, FORCING>(h, ph);
  // as in aa_node: the offsets of the stores are found anew
  typename St::T *out = buf;
  int ox = xw, oy = y, oz = z;
  asm volatile("" : "+l"(out), "+r"(ox), "+r"(oy), "+r"(oz));
  uint32_t *ow = reinterpret_cast<uint32_t *>(out);
  const int os = (oz * ny + oy) * wpr + ox;
  const auto half_at = [&](int row, int x, int p) {  // node x of row `row`
    return out + (pop_base<S, int>(row * 2 * wpr + x) + p * kBlockNodes);
  };
  if (!ODD) {
    // whole words: the slots of a solid node, which no node uses, stay zero
    if (skip_a && skip_b) return;
#pragma unroll
    for (int p = 0; p < kQ; ++p)
      ow[word(os) + opp(p) * kW] = P::pack(make_float2(skip_a ? 0.f : h[p].x, skip_b ? 0.f : h[p].y));
    return;
  }
  const int oym = wrap_m1(oy, ny), oyp = wrap_p1(oy, ny);
  const int ozm = wrap_m1(oz, g.nz), ozp = wrap_p1(oz, g.nz);
  const int xa = 2 * ox, xb = xa + 1;
#pragma unroll
  for (int p = 0; p < kQ; ++p) {
    const int ty = cy(p) == 1 ? oyp : (cy(p) == -1 ? oym : oy);
    const int tz = cz(p) == 1 ? ozp : (cz(p) == -1 ? ozm : oz);
    const int row = tz * ny + ty;
    const bool back_a = (bb.x >> opp(p)) & 1u, back_b = (bb.y >> opp(p)) & 1u;
    if (cx(p) == 0 && !(skip_a || skip_b || back_a || back_b)) {
      ow[word(row * wpr + ox) + p * kW] = P::pack(h[p]);
      continue;
    }
    if (!skip_a) {
      const int t = cx(p) == 1 ? wrap_p1(xa, nx) : (cx(p) == -1 ? wrap_m1(xa, nx) : xa);
      St::store(half_at(back_a ? oz * ny + oy : row, back_a ? xa : t, back_a ? opp(p) : p), h[p].x);
    }
    if (!skip_b) {
      const int t = cx(p) == 1 ? wrap_p1(xb, nx) : (cx(p) == -1 ? xa : xb);
      St::store(half_at(back_b ? oz * ny + oy : row, back_b ? xb : t, back_b ? opp(p) : p), h[p].y);
    }
  }
}

template <typename T2, int S, int FORCING, bool ODD>
__global__ void __launch_bounds__(32 * kRowsPerBlock, FORCING == kForcingNone ? 4 : 3)
    k_aa_stream_collide_pair(LbGeom g, LbPhys ph, typename Store<S>::T *buf, DevStatus *bump) {
  const int xw = blockIdx.x * 32 + threadIdx.x;
  const int y = blockIdx.y * kRowsPerBlock + threadIdx.y;
  const int z = blockIdx.z;
  if (bump != nullptr && xw == 0 && y == 0 && z == 0) bump->step += 1;
  if (xw >= (g.pitch >> 1) || y >= g.ny) return;
  aa_pair<T2, S, FORCING, ODD>(g, ph, buf, xw, y, z);
}

template <typename T2, int S, int FORCING>
void aa_pair_step(const LbGeom &g, const LbPhys &ph, void *buf, int odd, DevStatus *bump, cudaStream_t s) {
  using T = typename Store<S>::T;
  const dim3 block(32, kRowsPerBlock);
  const dim3 grid((g.pitch / 2 + 31) / 32, (g.ny + kRowsPerBlock - 1) / kRowsPerBlock, g.nz);
  if (odd)
    k_aa_stream_collide_pair<T2, S, FORCING, true><<<grid, block, 0, s>>>(g, ph, (T *)buf, bump);
  else
    k_aa_stream_collide_pair<T2, S, FORCING, false><<<grid, block, 0, s>>>(g, ph, (T *)buf, bump);
}
template <typename T2, int S>
cudaError_t aa_launch_pair(const LbGeom &g, const LbPhys &ph, void *buf, int odd, DevStatus *bump,
                           cudaStream_t s) {
  if (ph.g[0] == 0.f && ph.g[1] == 0.f && ph.g[2] == 0.f)
    aa_pair_step<T2, S, kForcingNone>(g, ph, buf, odd, bump, s);
  else if (ph.forcing == LBMD_FORCING_GUO)
    aa_pair_step<T2, S, LBMD_FORCING_GUO>(g, ph, buf, odd, bump, s);
  else
    aa_pair_step<T2, S, LBMD_FORCING_PAPER>(g, ph, buf, odd, bump, s);
  return cudaGetLastError();
}

template <int S, typename I, int NOISE>
cudaError_t aa_launch(const LbGeom &g, const LbPhys &ph, void *buf, int odd, DevStatus *bump,
                      cudaStream_t s) {
  using T = typename Store<S>::T;
  dim3 block(32, kRowsPerBlock);
  dim3 grid(g.ntx, (g.ny + kRowsPerBlock - 1) / kRowsPerBlock, g.nz);
  T *b = (T *)buf;
  const bool none = ph.g[0] == 0.f && ph.g[1] == 0.f && ph.g[2] == 0.f;
  if (odd) {
    if (none)
      k_aa_stream_collide<S, kForcingNone, I, true, NOISE><<<grid, block, 0, s>>>(g, ph, b, bump);
    else if (ph.forcing == LBMD_FORCING_GUO)
      k_aa_stream_collide<S, LBMD_FORCING_GUO, I, true, NOISE><<<grid, block, 0, s>>>(g, ph, b, bump);
    else
      k_aa_stream_collide<S, LBMD_FORCING_PAPER, I, true, NOISE><<<grid, block, 0, s>>>(g, ph, b, bump);
  } else {
    if (none)
      k_aa_stream_collide<S, kForcingNone, I, false, NOISE><<<grid, block, 0, s>>>(g, ph, b, bump);
    else if (ph.forcing == LBMD_FORCING_GUO)
      k_aa_stream_collide<S, LBMD_FORCING_GUO, I, false, NOISE><<<grid, block, 0, s>>>(g, ph, b, bump);
    else
      k_aa_stream_collide<S, LBMD_FORCING_PAPER, I, false, NOISE><<<grid, block, 0, s>>>(g, ph, b, bump);
  }
  return cudaGetLastError();
}

template <int NOISE>
cudaError_t aa_launch_f32(const LbGeom &g, const LbPhys &ph, void *buf, int odd, DevStatus *bump,
                          cudaStream_t s) {
  if ((long long)kQ * g.Vp < 0x7fffffffLL) return aa_launch<LBMD_STORE_F32, int, NOISE>(g, ph, buf, odd, bump, s);
  return aa_launch<LBMD_STORE_F32, size_t, NOISE>(g, ph, buf, odd, bump, s);
}

template <int NOISE>
cudaError_t aa_launch_storage(int storage, const LbGeom &g, const LbPhys &ph, void *buf, int odd,
                              DevStatus *bump, cudaStream_t s) {
  // 32-bit offsets when every population index fits
  const bool small = (long long)kQ * g.Vp < 0x7fffffffLL;
  // 16-bit storage: two nodes per thread except in narrow boxes (kNarrow), in the odd
  // step only in boxes of 2^17 nodes or more without a wall across x or of 192 nodes
  // or more in x (figures at aa_pair)
  if constexpr (NOISE == kNoNoise)
    if (small && g.pitch % 2 == 0 && g.nx > kNarrow &&
        (!odd || ((long long)g.nx * g.ny * g.nz >= 1 << 17 && (g.wall.wall_x < 0 || g.nx >= 192)))) {
      if (storage == LBMD_STORE_F16) return aa_launch_pair<__half2, LBMD_STORE_F16>(g, ph, buf, odd, bump, s);
      if (storage == LBMD_STORE_BF16)
        return aa_launch_pair<__nv_bfloat162, LBMD_STORE_BF16>(g, ph, buf, odd, bump, s);
    }
  switch (storage) {
    case LBMD_STORE_F32:
      return aa_launch_f32<NOISE>(g, ph, buf, odd, bump, s);
    case LBMD_STORE_F16:
      return small ? aa_launch<LBMD_STORE_F16, int, NOISE>(g, ph, buf, odd, bump, s)
                   : aa_launch<LBMD_STORE_F16, size_t, NOISE>(g, ph, buf, odd, bump, s);
    case LBMD_STORE_BF16:
      return small ? aa_launch<LBMD_STORE_BF16, int, NOISE>(g, ph, buf, odd, bump, s)
                   : aa_launch<LBMD_STORE_BF16, size_t, NOISE>(g, ph, buf, odd, bump, s);
  }
  return cudaErrorInvalidValue;
}

}  // namespace lbmd
