// lb_pull.cuh -- pull streaming with halfway bounce-back, shared by the
// stream-collide kernels, the read-out kernels and the bead gather.
#pragma once

#include "lbmd_common.cuh"

namespace lbmd {

// Row length of the populations of storage S (pad: see LbGeom::pitch).
template <int S>
__device__ __forceinline__ int row_pitch(const LbGeom &g) {
  return S == LBMD_STORE_F32 ? g.nx : g.pitch;
}
// Index of the population row-major order from that of the nodes.
template <int S, typename I>
__device__ __forceinline__ I pop_node(const LbGeom &g, I node) {
  if (S == LBMD_STORE_F32 || g.pitch == g.nx) return node;
  return node + (I)((unsigned)node / (unsigned)g.nx);  // one padding element per row
}

// Pre-collision deviations h_p(x, t+1) of node (x, y, z) from the
// post-collision buffer `src` (Eq. 5 free streaming, pull form):
//   h_p(x) = h*_p(x - c_p)      if x - c_p is fluid,
//   h_p(x) = h*_opp(p)(x)       otherwise (the population that left x towards
//                               the solid node comes back reversed),
// where bit p of `bb` says whether x - c_p is solid (the node's link mask; 0
// for a node known to be far from any solid node).  h*_q(y) sits at [q][y]
// (SWAP = false, kPopPull) or at [opp(q)][y] (SWAP = true, kPopAASwap).  I is
// the index type of the population offsets: int when 19 Vp < 2^31 (cheaper
// address arithmetic), size_t otherwise.
template <int S, typename I = size_t, bool SWAP = false>
__device__ __forceinline__ void pull19_mask(const LbGeom &g,
                                            const typename Store<S>::T *__restrict__ src, int x,
                                            int y, int z, uint32_t bb, float h[kQ]) {
  using St = Store<S>;
  const int nx = g.nx, ny = g.ny, nz = g.nz, pitch = row_pitch<S>(g);
  const int xm = wrap_m1(x, nx), xp = wrap_p1(x, nx);
  const int ym = wrap_m1(y, ny), yp = wrap_p1(y, ny);
  const int zm = wrap_m1(z, nz), zp = wrap_p1(z, nz);
  const I self = ((I)z * ny + y) * pitch + x;
  const I st = pop_stride<S, I>((I)g.Vp);
#pragma unroll
  for (int p = 0; p < kQ; ++p) {
    // source node x - c_p
    const int sx = cx(p) == 1 ? xm : (cx(p) == -1 ? xp : x);
    const int sy = cy(p) == 1 ? ym : (cy(p) == -1 ? yp : y);
    const int sz = cz(p) == 1 ? zm : (cz(p) == -1 ? zp : z);
    const I sidx = (I)(SWAP ? opp(p) : p) * st + pop_base<S, I>(((I)sz * ny + sy) * pitch + sx);
    const I bidx = (I)(SWAP ? p : opp(p)) * st + pop_base<S, I>(self);
    h[p] = St::load(src + (((bb >> p) & 1u) ? bidx : sidx));
  }
}

// Whether node (x, y) or, with W > 1, one of the W nodes from x on may have a
// solid node within one node: it is in or beside a wall layer or a solid row.
// (In the pore's opening such a node's link mask is zero.)
//
// Computed, so that the few nodes beside a wall read their mask word while the
// populations are on their way.  The stream-collides used to read a flag per
// 32-node tile and, in tiles next to a solid node, the mask before they could
// load a population (a quarter of the tiles of the 256x128x128 box with one
// wall layer, each waiting for two more memory latencies: FP32 100.4 us a step
// against 94.6 without the wall).  The mask itself is not computed: the bits of
// 18 directions cost the 16-bit kernel, bound by instructions, more than the
// load (70.7 us against 61.5).
template <int W = 1>
__device__ __forceinline__ bool beside_wall(const LbGeom &g, int x, int y) {
  const WallGeom &w = g.wall;
  int dx = x - w.wall_x;  // layers after the first one, around the box
  if (dx < 0) dx += g.nx;
  return (w.wall_x >= 0 && (dx <= w.wall_t || dx >= g.nx - W)) ||
         (w.y_walls && (y <= 1 || y >= g.ny - 2));
}

// The bounce-back of pull19_mask after the fact: h holds the values of every
// source x - c_p, solid or not; those of the solid ones (bits of `bb`) are
// replaced by the node's own reversed populations (self: its index in the
// populations' rows).
template <int S, typename I = size_t>
__device__ __forceinline__ void bounce19(const LbGeom &g, const typename Store<S>::T *__restrict__ src,
                                         I self, uint32_t bb, float h[kQ]) {
  using St = Store<S>;
  const I st = pop_stride<S, I>((I)g.Vp);
  const typename St::T *own = src + pop_base<S, I>(self);
#pragma unroll
  for (int p = 1; p < kQ; ++p)
    if ((bb >> p) & 1u) h[p] = St::load(own + (I)opp(p) * st);
}

__device__ __forceinline__ bool tile_is_near(const LbGeom &g, int x, int y, int z) {
  return __ldg(&g.tile_near[((size_t)z * g.ny + y) * g.ntx + (x >> 5)]) != 0;
}

// Pre-collision deviations h_p(x, t) of fluid node (x, y, z) for populations
// held in layout `mode` (kPop*), taking the link mask only where a solid node
// is within one node of the node's tile.  For read-outs and the bead gather,
// which run while no kernel writes `src` (gather_goes_first).
template <int S, typename I = size_t>
__device__ __forceinline__ void fetch19(const LbGeom &g, const typename Store<S>::T *__restrict__ src,
                                        int x, int y, int z, int mode, float h[kQ]) {
  using St = Store<S>;
  const I self = ((I)z * g.ny + y) * g.nx + x;
  if (mode == kPopAALocal) {
    const I own = ((I)z * g.ny + y) * row_pitch<S>(g) + x;
#pragma unroll
    for (int p = 0; p < kQ; ++p) h[p] = St::load(src + (I)p * pop_stride<S, I>((I)g.Vp) + pop_base<S, I>(own));
    return;
  }
  const uint32_t bb = tile_is_near(g, x, y, z) ? __ldg(&g.lmask[self]) : 0u;
  if (mode == kPopAASwap)
    pull19_mask<S, I, true>(g, src, x, y, z, bb, h);
  else
    pull19_mask<S, I, false>(g, src, x, y, z, bb, h);
}

// rho - rho0 and the momentum sum_p h_p c_p (sum_p w_p c_p = 0).
__device__ __forceinline__ void moments19(const float h[kQ], float &drho, float &jx, float &jy,
                                          float &jz) {
  drho = 0.f;
  jx = jy = jz = 0.f;
#pragma unroll
  for (int p = 0; p < kQ; ++p) {
    drho += h[p];
    if (cx(p)) jx += cx(p) > 0 ? h[p] : -h[p];
    if (cy(p)) jy += cy(p) > 0 ? h[p] : -h[p];
    if (cz(p)) jz += cz(p) > 0 ? h[p] : -h[p];
  }
}

}  // namespace lbmd
