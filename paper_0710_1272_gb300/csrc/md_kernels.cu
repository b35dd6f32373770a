// md_kernels.cu -- bead <-> fluid coupling and the constrained polymer MD cycle
// (arXiv:0710.1272, Sec. II: Eqs. 1-4, 10, the four-stage LB step; Sec. III:
// pulling force, wall, translocation bookkeeping).
//
// k_gather computes, for every (bead, corner) pair, the transfer weight and
// the fluid velocity of the pulled pre-collision populations, and sums them
// per bead (trilinear over the fluid corners, or nearest grid point).
// k_md_cycle then runs one thread block per chain, one thread per bead, and
// M substeps of
//     F = F_WCA + F_bend + F_wall + F_drive - m gamma (v - u_i) + F_r,
//     v += dt F / m,  r~ = r + dt v,
//     SHAKE: Newton on the N-1 bond multipliers, the tridiagonal Jacobian
//            solved by parallel cyclic reduction (TriPart),
//     v = (r' - r) / dt,  r = r',
//     RATTLE: one tridiagonal solve removes the bond-parallel relative
//             velocities,
//     J_i += dt (F_drag + F_r);
//   then the translocation bookkeeping.  The spread hands -J_i to the fluid
//   with the gather weights (Eq. 10 with the reaction sign): the gather claims
//   each transfer node for its smallest (bead, corner) entry, the impulses are
//   summed at that owner in 64-bit fixed point, and the owner adds the source
//   to the node's post-collision populations once -- so a step gives the same
//   bits whatever order the atomics take.
#include "lb_pull.cuh"

namespace lbmd {

constexpr float kTwoSixth = 1.122462048309373f;  // 2^(1/6)
constexpr float kSkin = 0.8f;  // neighbour-list skin: lists hold pairs within r_c + skin

// How the pair and wall forces of a chain are found (DevStatus::nl_ok).
constexpr int kNlNone = 0;  // a bead's list overflowed: all pairs, stencil scan
constexpr int kNlBead = 1;  // per-bead lists in the workspace
constexpr int kNlFlat = 2;  // one list of (bead, partner) entries in shared memory

struct F3 {
  float x, y, z;
};
__device__ __forceinline__ F3 f3(float4 v) { return F3{v.x, v.y, v.z}; }
__device__ __forceinline__ float4 f4(F3 v) { return make_float4(v.x, v.y, v.z, 0.f); }
__device__ __forceinline__ F3 operator+(F3 a, F3 b) { return F3{a.x + b.x, a.y + b.y, a.z + b.z}; }
__device__ __forceinline__ F3 operator-(F3 a, F3 b) { return F3{a.x - b.x, a.y - b.y, a.z - b.z}; }
__device__ __forceinline__ F3 operator*(float s, F3 a) { return F3{s * a.x, s * a.y, s * a.z}; }
// a . b with its roundings written out: which product of a sum is rounded and
// which is fused is the compiler's choice otherwise, and a chain's bits with it
// (chains of stiff beads, and any in 16-bit populations, carry a different last
// bit into the fifth digit of the velocities within twenty steps).
__device__ __forceinline__ float dot(F3 a, F3 b) {
  return __fmaf_rn(a.z, b.z, __fmaf_rn(a.x, b.x, __fmul_rn(a.y, b.y)));
}
__device__ __forceinline__ float dot_yx(F3 a, F3 b) {
  return __fmaf_rn(a.z, b.z, __fmaf_rn(a.y, b.y, __fmul_rn(a.x, b.x)));
}

// Threads of the MD block: one per bead in whole warps; for chains of up to 224
// beads warps that only evaluate the force list, beside the bead warps' own work
// (two for up to 32 beads, four for up to 96, else eight: 40 beads 28.9 us a step
// with four, 30.3 with eight; 100 beads 34.7 and 34.3; 128 beads 37.3 and 35.9);
// and for chains of more than two warps one more for the boundary system of the
// tridiagonal solves, where the block's register class (512, 768, 896 or 1024
// threads: 128, 80, 72 or 64 registers) has room for it, else warp 0 solves it
// (four chains of 40 beads 34.1 us a step, 34.8 with a warp of its own).
__host__ __device__ inline int bead_threads(int N) { return (N + 31) / 32 * 32; }
int md_threads(int N) {
  int t = bead_threads(N);
  if (t <= 32) return t + 64;
  const bool two = t == 64;
  if (t <= 224) t += t <= 96 ? 128 : 256;
  return two || t == 512 || t == 768 || t == 896 || t == LBMD_MAX_BEADS ? t : t + 32;
}
// The block of an ensemble's chains: sizes in steps of 64 threads up to 512,
// then the register classes, so that few launches take chains of every length
// (nine at most; the warps to spare evaluate the force list), and small, so that
// several chains share an SM and leave registers to the stream-collide.
int md_group_threads(int N) {
  const int b = bead_threads(N) < 96 ? 96 : bead_threads(N);
  const int t = b == 512 || b == 768 || b == LBMD_MAX_BEADS ? b : b + 32;
  return t <= 512 ? (t + 63) / 64 * 64 : t <= 768 ? 768 : LBMD_MAX_BEADS;
}

// Shared memory of the MD block: per bead positions (hi, lo), displacements,
// bond vectors at the start and the end of the substep, multipliers and the
// mask of acting list entries; then the force list (8 bytes an entry) and a
// separation and force factor per entry, eight entries per bead (the chains
// measured average three) and 128 for the beads in the pore, as far as 220 KB
// reach.
constexpr int kMdSmemMost = 220000;
constexpr size_t kSmemOfBlock = 227 * 1024;  // the most that one block may have
__host__ __device__ inline size_t md_smem_head(int N) {
  return ((size_t)N * (5 * sizeof(float4) + 2 * sizeof(float)) + 15) / 16 * 16;
}
__host__ __device__ inline int item_want(int N) { return 8 * N + 128; }
__host__ __device__ inline int item_cap(int N) {
  const int room = (kMdSmemMost - (int)md_smem_head(N)) / (int)(sizeof(float4) + sizeof(uint2));
  return item_want(N) < room ? item_want(N) : room;
}
int md_item_cap(int N) { return item_cap(N); }
// Never less for a longer chain (an ensemble sizes a group's blocks for its
// longest one): chains whose list is cut to the room there is ask for all of it.
size_t md_smem_bytes(int N) {
  if (item_cap(N) < item_want(N)) return kMdSmemMost;
  return md_smem_head(N) + (size_t)item_cap(N) * (sizeof(float4) + sizeof(uint2));
}

// Double-float helpers: a coordinate is hi + lo with |lo| <= ulp(hi) / 2.
__device__ __forceinline__ void two_sum_add(float &hi, float &lo, float d) {
  const float s = hi + d;
  const float bp = s - hi;
  const float e = (hi - (s - bp)) + (d - bp);
  const float l = lo + e;
  hi = s + l;
  lo = l - (hi - s);
}
__device__ __forceinline__ F3 diff_hl(float4 ah, float4 al, float4 bh, float4 bl) {
  return F3{(ah.x - bh.x) + (al.x - bl.x), (ah.y - bh.y) + (al.y - bl.y),
            (ah.z - bh.z) + (al.z - bl.z)};
}
// Index into [0, n): one add or subtract for indices within a period of the
// box (the common case), the integer remainder otherwise.
__device__ __forceinline__ int wrap_near(int a, int n) {
  if (a < 0) a += n;
  if (a >= n) a -= n;
  if ((unsigned)a >= (unsigned)n) a = wrapi(a, n);
  return a;
}

// Wrapped node index and fraction of global = origin + hi + lo.
__device__ __forceinline__ void cell_frac_hl(float hi, float lo, int origin, int n, int &cell,
                                             float &frac) {
  const float fl = floorf(hi);
  frac = (hi - fl) + lo;
  cell = wrap_near(origin + (int)fl, n);
}

// 2x2 matrices for the interface system of the tridiagonal solve.
struct M2 {
  float a, b, c, d;  // [[a, b], [c, d]]
};
__device__ __forceinline__ M2 mmul(M2 x, M2 y) {
  return M2{x.a * y.a + x.b * y.c, x.a * y.b + x.b * y.d, x.c * y.a + x.d * y.c,
            x.c * y.b + x.d * y.d};
}
__device__ __forceinline__ M2 madd(M2 x, M2 y) { return M2{x.a + y.a, x.b + y.b, x.c + y.c, x.d + y.d}; }

// Hardware reciprocal approximation (relative error ~2^-23) for the
// tridiagonal solves: they are latency-bound chains, and a correctly rounded
// reciprocal costs several dependent instructions.
__device__ __forceinline__ float rcp_fast(float x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}

__device__ __forceinline__ M2 minv(M2 x) {
  const float r = rcp_fast(x.a * x.d - x.b * x.c);
  return M2{x.d * r, -x.b * r, -x.c * r, x.a * r};
}
__device__ __forceinline__ M2 mshfl_up(M2 x, int s) {
  return M2{__shfl_up_sync(0xffffffffu, x.a, s), __shfl_up_sync(0xffffffffu, x.b, s),
            __shfl_up_sync(0xffffffffu, x.c, s), __shfl_up_sync(0xffffffffu, x.d, s)};
}
__device__ __forceinline__ M2 mshfl_down(M2 x, int s) {
  return M2{__shfl_down_sync(0xffffffffu, x.a, s), __shfl_down_sync(0xffffffffu, x.b, s),
            __shfl_down_sync(0xffffffffu, x.c, s), __shfl_down_sync(0xffffffffu, x.d, s)};
}


// s a + b, each component one fused operation.
__device__ __forceinline__ F3 axpy(float s, F3 a, F3 b) {
  return F3{fmaf(s, a.x, b.x), fmaf(s, a.y, b.y), fmaf(s, a.z, b.z)};
}

// Barriers of a part of the block: the warps that hold beads, with or without
// the warp that solves the boundary system.  `threads` counts all that take
// part; every one of them meets the same barriers in the same order, whole
// warps at a time.
constexpr int kBarBeads = 1, kBarVote = 2, kBarSides = 3, kBarMiddle = 4;
__device__ __forceinline__ void bar_sync(int id, int threads) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}
__device__ __forceinline__ void bar_arrive(int id, int threads) {
  asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(threads) : "memory");
}
__device__ __forceinline__ bool bar_all(int id, int threads, bool p) {
  int r;
  asm volatile(
      "{\n\t.reg .pred q, o;\n\tsetp.ne.s32 q, %3, 0;\n\tbar.red.and.pred o, %1, %2, q;\n\t"
      "selp.s32 %0, 1, 0, o;\n\t}"
      : "=r"(r)
      : "r"(id), "r"(threads), "r"((int)p)
      : "memory");
  return r != 0;
}

// Tridiagonal solve over rows 0..n-1 (row i held by thread i: a x_{i-1} + b x_i
// + c x_{i+1} = d, with a_0 = c_{n-1} = 0), SPIKE-type partition by warps: each
// warp reduces its 32 rows by cyclic reduction over lane shuffles, for the
// right-hand side and for the two coupling columns to the neighbouring warps
// (the "spikes" v and w), giving x_i = y_i - v_i x_last(prev warp) - w_i
// x_first(next warp) (tri_reduce).  The first and last unknowns of neighbouring
// warps form a block tridiagonal system with 2x2 blocks, one block row per warp
// boundary, which one warp solves by block cyclic reduction (tri_boundary).
// Rows past the chain are identity rows.
//
// What bounds it is latency, and the shuffles of many warps.  A partition over
// the lanes of a single warp, with the rows in registers, is faster (400 rows
// 1.1 k cycles; this one 2.9 k, sides 0.9 k and boundaries 2.0 k), but its last
// bits differ, and with them the trajectories (see dot).
struct TriPart {
  float y, v, w;
};
// SPIKES: the chain has more than one warp.  Before round s the columns r1 and
// r2 are zero but in the first and the last s lanes, so of each only one
// neighbour counts.
template <bool SPIKES>
__device__ __forceinline__ TriPart tri_reduce(int n, float a, float b, float c, float d) {
  const int t = threadIdx.x, lane = t & 31;
  if (t >= n) {
    a = 0.f;
    b = 1.f;
    c = 0.f;
    d = 0.f;
  }
  float al = lane == 0 ? 0.f : a, be = b, ga = lane == 31 ? 0.f : c;
  float r0 = d, r1 = lane == 0 ? a : 0.f, r2 = lane == 31 ? c : 0.f;
#pragma unroll
  for (int s = 1; s < 32; s <<= 1) {
    const float bm = __shfl_up_sync(0xffffffffu, be, s), bp = __shfl_down_sync(0xffffffffu, be, s);
    const float gm = __shfl_up_sync(0xffffffffu, ga, s), ap = __shfl_down_sync(0xffffffffu, al, s);
    const float r0m = __shfl_up_sync(0xffffffffu, r0, s), r0p = __shfl_down_sync(0xffffffffu, r0, s);
    const bool hm = lane >= s, hp = lane + s < 32;
    const float k1 = hm ? al * rcp_fast(bm) : 0.f;
    const float k2 = hp ? ga * rcp_fast(bp) : 0.f;
    if (SPIKES) {
      r1 = __fmaf_rn(-k1, __shfl_up_sync(0xffffffffu, r1, s), r1);
      r2 = __fmaf_rn(-k2, __shfl_down_sync(0xffffffffu, r2, s), r2);
    }
    if (s < 16) {
      const float am = __shfl_up_sync(0xffffffffu, al, s), gp = __shfl_down_sync(0xffffffffu, ga, s);
      al = hm ? -k1 * am : 0.f;
      ga = hp ? -k2 * gp : 0.f;
    }
    be = __fmaf_rn(-k2, ap, __fmaf_rn(-k1, gm, be));
    r0 = __fmaf_rn(-k2, r0p, __fmaf_rn(-k1, r0m, r0));
  }
  const float ib = rcp_fast(be);
  return TriPart{r0 * ib, r1 * ib, r2 * ib};
}
// The system of the nch - 1 boundaries between nch warps: from the parts of
// each warp's first and last row (s_y, six floats a warp) the unknowns of the
// last row [0, 32) and the first row [32, 64) of each warp.  By one warp.
__device__ __forceinline__ void tri_boundary(int nch, const float *s_y, float *s_x) {
  const int lane = threadIdx.x & 31;
  // block row k: unknowns (x_last(k), x_first(k+1)) at the boundary of
  // warps k and k+1; rows beyond nch-2 are identity rows
  M2 L{0.f, 0.f, 0.f, 0.f}, D{1.f, 0.f, 0.f, 1.f}, U{0.f, 0.f, 0.f, 0.f};
  float q0 = 0.f, q1 = 0.f;
  if (lane < nch - 1) {
    D.b = s_y[6 * lane + 5];        // w of the last row of warp k
    D.c = s_y[6 * (lane + 1) + 1];  // v of the first row of warp k+1
    L.a = s_y[6 * lane + 4];        // v of the last row of warp k
    U.d = s_y[6 * (lane + 1) + 2];  // w of the first row of warp k+1
    q0 = s_y[6 * lane + 3];
    q1 = s_y[6 * (lane + 1)];
  }
  // block cyclic reduction over the nch - 1 boundary rows; each lane
  // inverts its own diagonal block and the neighbours' inverses arrive by
  // shuffle
  for (int s = 1; s < nch - 1; s <<= 1) {
    const M2 Di = minv(D);
    const M2 Lm = mshfl_up(L, s), Dim = mshfl_up(Di, s), Um = mshfl_up(U, s);
    const float q0m = __shfl_up_sync(0xffffffffu, q0, s), q1m = __shfl_up_sync(0xffffffffu, q1, s);
    const M2 Lp = mshfl_down(L, s), Dip = mshfl_down(Di, s), Up = mshfl_down(U, s);
    const float q0p = __shfl_down_sync(0xffffffffu, q0, s), q1p = __shfl_down_sync(0xffffffffu, q1, s);
    M2 al2{0.f, 0.f, 0.f, 0.f}, ga2{0.f, 0.f, 0.f, 0.f};
    if (lane >= s) {
      const M2 t2 = mmul(L, Dim);
      al2 = M2{-t2.a, -t2.b, -t2.c, -t2.d};
    }
    if (lane + s < 32) {
      const M2 t2 = mmul(U, Dip);
      ga2 = M2{-t2.a, -t2.b, -t2.c, -t2.d};
    }
    const M2 nL = mmul(al2, Lm), nU = mmul(ga2, Up);
    D = madd(D, madd(mmul(al2, Um), mmul(ga2, Lp)));
    const float nq0 = q0 + al2.a * q0m + al2.b * q1m + ga2.a * q0p + ga2.b * q1p;
    const float nq1 = q1 + al2.c * q0m + al2.d * q1m + ga2.c * q0p + ga2.d * q1p;
    L = nL;
    U = nU;
    q0 = nq0;
    q1 = nq1;
  }
  const M2 Di = minv(D);
  if (lane < nch - 1) {
    s_x[lane] = Di.a * q0 + Di.b * q1;           // x_last of warp k
    s_x[32 + lane + 1] = Di.c * q0 + Di.d * q1;  // x_first of warp k+1
  }
}
// The unknown of a row of warp w from its part and the boundaries' unknowns.
__device__ __forceinline__ float tri_finish(TriPart t, int w, int nch, const float *s_x) {
  float x = t.y;
  if (w > 0) x -= t.v * s_x[w - 1];
  if (w + 1 < nch) x -= t.w * s_x[32 + w + 1];
  return x;
}

// Eq. 2 truncated at 2^(1/6) sigma: adds -dV/dd for separation d.
__device__ __forceinline__ void wca_add(F3 d, float sig2, float rc2, float eps24, F3 &F) {
  const float r2 = dot(d, d);
  if (r2 < rc2) {
    const float ir2 = 1.0f / r2;
    const float sr2 = sig2 * ir2;
    const float sr6 = sr2 * sr2 * sr2;
    const float f = eps24 * (2.0f * sr6 * sr6 - sr6) * ir2;
    F = F + f * d;
  }
}

// Eq. 3 bending at the angle of beads (a, b, c) given the two bond vectors
// b1 = r_b - r_a and b2 = r_c - r_b, their lengths and product: with
// V = kappa phi^2 / 2 the forces F = -dV/dr on a, b and c are -A g1, A (g1 - g2)
// and A g2; returns A.
__device__ __forceinline__ float bend_terms(F3 b1, F3 b2, float l1, float l2, float b12, float kappa, F3 &g1,
                                         F3 &g2) {
  const float cphi = fminf(1.f, fmaxf(-1.f, b12 / (l1 * l2)));
  const float phi = acosf(cphi);
  const float A = phi < 1e-4f ? kappa : kappa * phi / sinf(phi);
  const float p = 1.0f / (l1 * l2), q1 = -(cphi / (l1 * l1)), q2 = -(cphi / (l2 * l2));
  g1 = axpy(q1, b1, F3{__fmul_rn(p, b2.x), __fmul_rn(p, b2.y), __fmul_rn(p, b2.z)});
  g2 = axpy(q2, b2, F3{__fmul_rn(p, b1.x), __fmul_rn(p, b1.y), __fmul_rn(p, b1.z)});
  return A;
}

// WCA pair forces on bead i from every other non-bonded bead (minimum image).
__device__ __noinline__ F3 all_pair_forces(const ChainArgs &a, int i, float4 rh, float4 rl,
                                              const float4 *s_rh, const float4 *s_rl) {
  const LbGeom &g = a.geo;
  const float sig2 = a.sigma * a.sigma;
  const float rc = kTwoSixth * a.sigma, rc2 = rc * rc;
  const float eps24 = 24.0f * a.eps;
  const float Lx = (float)g.nx, Ly = (float)g.ny, Lz = (float)g.nz;
  const float iLx = 1.0f / Lx, iLy = 1.0f / Ly, iLz = 1.0f / Lz;
  F3 F{0.f, 0.f, 0.f};
  for (int j = 0; j < a.N; ++j) {
    const int dij = j - i;
    if (dij == 0 || (a.has_bonds && (dij == 1 || dij == -1))) continue;
    F3 d = diff_hl(rh, rl, s_rh[j], s_rl[j]);
    d.x -= Lx * rintf(d.x * iLx);
    d.y -= Ly * rintf(d.y * iLy);
    d.z -= Lz * rintf(d.z * iLz);
    wca_add(d, sig2, rc2, eps24, F);
  }
  return F;
}

// Sec. III pulling force on a bead at the local position rh + rl: -f_drive x
// inside the channel of the pore cross-section and the x-layers within 1.5
// nodes of the wall.
__device__ __forceinline__ F3 drive_force_at(const ChainArgs &a, float4 rh, float4 rl) {
  const LbGeom &g = a.geo;
  F3 F{0.f, 0.f, 0.f};
  if (a.has_wall && a.pore_d > 0 && a.fdrive != 0.f) {
    int c[3];
    float sf[3];
    cell_frac_hl(rh.x, rl.x, a.ox, g.nx, c[0], sf[0]);
    cell_frac_hl(rh.y, rl.y, a.oy, g.ny, c[1], sf[1]);
    cell_frac_hl(rh.z, rl.z, a.oz, g.nz, c[2], sf[2]);
    const int di = wrap_near(c[0] - a.wall_x + g.nx / 2, g.nx) - g.nx / 2;
    const float dx = (float)di + sf[0] - 0.5f * (float)(a.wall_t - 1);
    const float half = 0.5f * (float)(a.wall_t - 1) + 1.5f;
    const float ry = (float)c[1] + sf[1], rz = (float)c[2] + sf[2];
    if (fabsf(dx) <= half && ry >= a.pore_y0 - 0.5f && ry < a.pore_y0 + a.pore_d - 0.5f &&
        rz >= a.pore_z0 - 0.5f && rz < a.pore_z0 + a.pore_d - 0.5f)
      F.x -= a.fdrive;
  }
  return F;
}

// Sum of K values over the block (every thread gets the sums).  red holds
// 32 K partials and K results; a result is rewritten only after every thread
// has passed the next call's first barrier, i.e. has read it.
template <int K>
__device__ __forceinline__ void block_sum(float (&v)[K], float *red) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
#pragma unroll
  for (int k = 0; k < K; ++k)
    for (int m = 16; m > 0; m >>= 1) v[k] += __shfl_xor_sync(0xffffffffu, v[k], m);
  if (lane == 0)
#pragma unroll
    for (int k = 0; k < K; ++k) red[warp * K + k] = v[k];
  __syncthreads();
  if (warp == 0) {
#pragma unroll
    for (int k = 0; k < K; ++k) {
      float t = lane < nw ? red[lane * K + k] : 0.f;
      for (int m = 16; m > 0; m >>= 1) t += __shfl_xor_sync(0xffffffffu, t, m);
      if (lane == 0) red[32 * K + k] = t;
    }
  }
  __syncthreads();
#pragma unroll
  for (int k = 0; k < K; ++k) v[k] = red[32 * K + k];
}

// Solid nodes around a bead within `radius` (node offsets n with
// |n - s| < radius per axis), from the Sec. III geometry itself (the wall layers
// minus the pore, and the rows y = 0 and y = ny - 1 with y-walls): the rule the
// solid bitfield is built from, with no memory read.  For each solid node calls
// fn(node coordinate in the chain's local frame).
//
// Two things once made it 56-73 k, then 36 k cycles a list build (N = 20 to
// 700), now 12 k.  Stepping through the x offsets had the lanes of a
// warp reach the wall's layer at different steps, one scan of it behind the
// other: without y-walls each layer is looked up.  And `a` may live in kernel
// parameters read through a pointer here, again after every store of fn: all
// that is needed of it is copied first.
template <typename Fn>
__device__ __forceinline__ void for_solid_nodes(const ChainArgs &a, float4 rh, float4 rl,
                                                float radius, Fn fn) {
  const int nx = a.geo.nx, ny = a.geo.ny, nz = a.geo.nz, wall_x = a.wall_x, wall_t = a.wall_t;
  const int py0 = a.pore_y0, pz0 = a.pore_z0, pd = a.pore_d, oy0 = a.oy, oz0 = a.oz;
  const bool has_wall = a.has_wall, y_walls = a.y_walls;
  if (!has_wall && !y_walls) return;
  int cx0, cy0 = 0, cz0 = 0;
  float sx, sy = 0.f, sz = 0.f;
  cell_frac_hl(rh.x, rl.x, a.ox, nx, cx0, sx);
  const int lo0 = (int)ceilf(sx - radius), hi0 = (int)floorf(sx + radius);
  const float fx = floorf(rh.x), fy = floorf(rh.y), fz = floorf(rh.z);
  // each layer is met at one offset where the box is wider than the stencil
  const bool layers = !y_walls && nx > 2 * ((int)radius + 2) + wall_t;
  const int steps = layers ? wall_t : hi0 - lo0 + 1;
  bool ready = false;
  int lo1 = 0, hi1 = 0, lo2 = 0, hi2 = 0;
  for (int k = 0; k < steps; ++k) {
    int ox = lo0 + k;
    if (layers) {
      ox = wall_x + k - cx0;
      if (ox < lo0) ox += nx;
      if (ox > hi0) ox -= nx;
      if (ox < lo0 || ox > hi0) continue;
    }
    int dx = wrap_near(cx0 + ox, nx) - wall_x;
    if (dx < 0) dx += nx;
    const bool layer = has_wall && dx < wall_t;
    if (!y_walls && !layer) continue;  // no solid node in this layer
    if (!ready) {  // few beads get here
      ready = true;
      cell_frac_hl(rh.y, rl.y, oy0, ny, cy0, sy);
      cell_frac_hl(rh.z, rl.z, oz0, nz, cz0, sz);
      lo1 = (int)ceilf(sy - radius), hi1 = (int)floorf(sy + radius);
      lo2 = (int)ceilf(sz - radius), hi2 = (int)floorf(sz + radius);
    }
    for (int oy = lo1; oy <= hi1; ++oy) {
      const int y = wrap_near(cy0 + oy, ny);
      const bool row = y_walls && (y == 0 || y == ny - 1);
      const bool open_y = pd > 0 && y >= py0 && y < py0 + pd;
      if (!row && !layer) continue;
      for (int oz = lo2; oz <= hi2; ++oz) {
        const int z = wrap_near(cz0 + oz, nz);
        if (!row && open_y && z >= pz0 && z < pz0 + pd) continue;  // the pore
        fn(make_float4(fx + (float)ox, fy + (float)oy, fz + (float)oz, 0.f));
      }
    }
  }
}

// Eq. 2 between the bead and a solid node given in the local frame.
__device__ __forceinline__ void wall_add(float4 rh, float4 rl, float4 node, float sig2, float rc2,
                                         float eps24, F3 &F) {
  wca_add(F3{(rh.x - node.x) + rl.x, (rh.y - node.y) + rl.y, (rh.z - node.z) + rl.z}, sig2, rc2,
          eps24, F);
}

// The minimum image of a separation.
__device__ __noinline__ F3 min_image(const LbGeom &g, F3 d) {
  const float Lx = (float)g.nx, Ly = (float)g.ny, Lz = (float)g.nz;
  d.x -= Lx * rintf(d.x * (1.0f / Lx));
  d.y -= Ly * rintf(d.y * (1.0f / Ly));
  d.z -= Lz * rintf(d.z * (1.0f / Lz));
  return d;
}

// Bead i's pair and wall forces from its own lists in the workspace
// (kNlBead).
__device__ __noinline__ F3 list_forces(const ChainArgs &a, int i, float4 rh, float4 rl,
                                          const float4 *s_rh, const float4 *s_rl) {
  const float sig2 = a.sigma * a.sigma;
  const float rc = kTwoSixth * a.sigma, rc2 = rc * rc;
  const float eps24 = 24.0f * a.eps;
  F3 F{0.f, 0.f, 0.f};
  const int np = a.nl_cnt[i], nw = a.wl_cnt[i];
  const short *L = a.nl_list + (size_t)i * kMaxPairs;
  for (int q = 0; q < np; ++q) {
    const int j = L[q] & (LBMD_MAX_BEADS - 1);
    wca_add(min_image(a.geo, diff_hl(rh, rl, s_rh[j], s_rl[j])), sig2, rc2, eps24, F);
  }
  const float4 *W = a.wl_list + (size_t)i * kMaxWall;
#pragma unroll 4
  for (int q = 0; q < nw; ++q) wall_add(rh, rl, W[q], sig2, rc2, eps24, F);
  return F;
}

// An entry of the flat force list: a bead and its partner, another bead or a
// solid node, in 64 bits -- x: bead (10 bits), the entry's number among the
// bead's own (5 bits, kItemTail from there on), kItemWall, and the node's x
// coordinate in the upper half; y: the partner bead | kItemImage, or the
// node's y and z coordinates (16-bit integers of the chain's local frame).
constexpr unsigned kItemTail = 31u;        // summed whether it acts or not
constexpr unsigned kItemWall = 1u << 15;   // partner is a solid node
constexpr unsigned kItemImage = 1u << 10;  // the pair reaches across a periodic boundary
constexpr short kPairImage = 1 << 14;      // the same in a bead's pair list
__device__ __forceinline__ bool fits_short(float4 n) {
  return fabsf(n.x) <= 32000.f && fabsf(n.y) <= 32000.f && fabsf(n.z) <= 32000.f;
}

// Evaluates the flat list: `who` of `of` threads share the entries.  An entry
// within the cutoff leaves its separation d and the factor f of its force f d in
// s_f (the bead adds f d by fused operations, as a walk along its own list
// does) and a bit in its bead's mask (the entry's number among the bead's own);
// integer ORs commute, so the result does not depend on the order of the threads.
//
// With a list per bead the chain waited for its fullest one (a bead in the
// pore: ~25 entries at ~200-290 cycles each, 3.5-5 k cycles of every substep).
// Spread over the block, two entries at a time and without a branch on the
// cutoff, whose latencies would follow one another (400 beads: 2.7 k cycles with
// the branch, 1.6 k without; 20 beads 1.3 and 0.8 k, with an approximate
// reciprocal in place of the division on both sides).
__device__ __forceinline__ void eval_items(const ChainArgs &a, const uint2 *s_item, int n, int who,
                                           int of, const float4 *s_rh, const float4 *s_rl, float4 *s_f,
                                           unsigned *s_mask) {
  const float sig2 = a.sigma * a.sigma;
  const float rc = kTwoSixth * a.sigma, rc2 = rc * rc;
  const float eps24 = 24.0f * a.eps;
#pragma unroll 1
  for (int q0 = who; q0 < n; q0 += 2 * of) {
    uint2 it[2];
    float4 rh[2], rl[2], oh[2], ol[2];
    it[0] = s_item[q0];
    it[1] = s_item[min(q0 + of, n - 1)];
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      const int i = it[k].x & (LBMD_MAX_BEADS - 1);
      const int j = (it[k].x & kItemWall) ? i : (int)(it[k].y & (LBMD_MAX_BEADS - 1));
      rh[k] = s_rh[i];
      rl[k] = s_rl[i];
      oh[k] = s_rh[j];
      ol[k] = s_rl[j];
    }
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      const int q = q0 + k * of;
      const bool wall = (it[k].x & kItemWall) != 0, tail = (it[k].x >> 10 & 31u) == kItemTail;
      const bool image = !wall && (it[k].y & kItemImage) != 0;
      if (wall) {
        oh[k] = make_float4((float)((int)it[k].x >> 16), (float)(short)(it[k].y & 0xffffu),
                            (float)((int)it[k].y >> 16), 0.f);
        ol[k] = make_float4(0.f, 0.f, 0.f, 0.f);
      }
      F3 d = diff_hl(rh[k], rl[k], oh[k], ol[k]);
      if (image) d = min_image(a.geo, d);
      const float r2 = dot(d, d);
      const bool in = q < n && r2 < rc2;
      const float ir2 = 1.0f / r2;
      const float sr2 = sig2 * ir2;
      const float sr6 = sr2 * sr2 * sr2;
      const float f = eps24 * (2.0f * sr6 * sr6 - sr6) * ir2;
      if (in || (tail && q < n)) s_f[q] = in ? make_float4(d.x, d.y, d.z, f) : make_float4(0.f, 0.f, 0.f, 0.f);
      if (in && !tail) atomicOr(&s_mask[it[k].x & (LBMD_MAX_BEADS - 1)], 1u << (it[k].x >> 10 & 31u));
    }
  }
}

// Rebuild the lists of bead i (thread i; called by the whole block, `bead`
// false for threads without one) with cutoff r_c + skin, in the workspace: the
// bead's pairs and solid nodes, and from them the flat list, which goes to
// shared memory as well.  Solid nodes are kept within the sphere of radius
// r_c + skin (a node beyond it exerts no force while the bead stays within
// half the skin of the build position).  Returns the kind of list that holds
// (kNl*), the same on every thread; *n_items entries of the flat one, of which
// *cnt from s_first[i] on are the bead's.
//
// The chain is walked in groups of 32 consecutive beads, which lie close
// together: a warp passes over a group whose bounding box is beyond the
// cutoff of all its beads, and tests the others branch-free into a bit mask,
// whose few set bits are then appended in bead order.
__device__ __noinline__ int build_lists(const ChainArgs &a, int i, bool bead, float4 rh, float4 rl,
                           const float4 *s_rh, const float4 *s_rl, uint2 *s_item, int *s_first,
                           int *n_items, int *cnt) {
  __shared__ float s_box[32][8];  // per group: centre and half extents (x, y, z)
  __shared__ int s_sum[32];
  const LbGeom &g = a.geo;
  const int N = a.N, groups = (N + 31) >> 5, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const float rlist = kTwoSixth * a.sigma + kSkin, rl2 = rlist * rlist;
  const float Lx = (float)g.nx, Ly = (float)g.ny, Lz = (float)g.nz;
  const float iLx = 1.0f / Lx, iLy = 1.0f / Ly, iLz = 1.0f / Lz;
  {
    const float big = 3.0e38f;
    F3 lo = bead ? f3(rh) : F3{big, big, big}, hi = bead ? f3(rh) : F3{-big, -big, -big};
#pragma unroll
    for (int m = 16; m > 0; m >>= 1) {
      lo.x = fminf(lo.x, __shfl_xor_sync(0xffffffffu, lo.x, m));
      lo.y = fminf(lo.y, __shfl_xor_sync(0xffffffffu, lo.y, m));
      lo.z = fminf(lo.z, __shfl_xor_sync(0xffffffffu, lo.z, m));
      hi.x = fmaxf(hi.x, __shfl_xor_sync(0xffffffffu, hi.x, m));
      hi.y = fmaxf(hi.y, __shfl_xor_sync(0xffffffffu, hi.y, m));
      hi.z = fmaxf(hi.z, __shfl_xor_sync(0xffffffffu, hi.z, m));
    }
    if (lane == 0 && warp < groups) {
      float *b = s_box[warp];
      b[0] = 0.5f * (lo.x + hi.x);
      b[1] = 0.5f * (lo.y + hi.y);
      b[2] = 0.5f * (lo.z + hi.z);
      b[3] = 0.5f * (hi.x - lo.x);
      b[4] = 0.5f * (hi.y - lo.y);
      b[5] = 0.5f * (hi.z - lo.z);
    }
  }
  __syncthreads();
  short *G = a.nl_list + (size_t)i * kMaxPairs;
  float4 *W = a.wl_list + (size_t)i * kMaxWall;
  uint2 *items = a.items;
  const int reach = a.has_bonds ? 1 : 0;
  int np = 0, nw = 0;
  // a pair of the list moves by at most two half skins until the next
  // rebuild: within this box width it keeps the image it has now
  const float room = 2.02f * (rlist + kSkin);
  const bool small = !(Lx > room && Ly > room && Lz > room);
  if (warp < groups) {
    for (int c = 0; c < groups; ++c) {
      const float *b = s_box[c];
      float ax = rh.x - b[0], ay = rh.y - b[1], az = rh.z - b[2];
      ax = fmaxf(fabsf(ax - Lx * rintf(ax * iLx)) - b[3], 0.f);
      ay = fmaxf(fabsf(ay - Ly * rintf(ay * iLy)) - b[4], 0.f);
      az = fmaxf(fabsf(az - Lz * rintf(az * iLz)) - b[5], 0.f);
      // beyond the cutoff with room for rounding; a NaN goes on to the test
      const bool far = !bead || ax * ax + ay * ay + az * az > 1.01f * rl2 + 0.01f;
      if (__all_sync(0xffffffffu, far)) continue;
      const int j0 = c << 5, nj = min(32, N - j0);
      unsigned mask = 0u;
#pragma unroll 4
      for (int jj = 0; jj < nj; ++jj) {
        F3 d = diff_hl(rh, rl, s_rh[j0 + jj], s_rl[j0 + jj]);
        d.x -= Lx * rintf(d.x * iLx);
        d.y -= Ly * rintf(d.y * iLy);
        d.z -= Lz * rintf(d.z * iLz);
        if (dot(d, d) < rl2) mask |= 1u << jj;
      }
      // not the bead itself, nor its bonded neighbours
      const int own = i - j0;
      for (int k = own - reach; k <= own + reach; ++k)
        if (k >= 0 && k < 32) mask &= ~(1u << k);
      if (!bead) mask = 0u;
      while (mask) {
        const int j = j0 + __ffs(mask) - 1;
        mask &= mask - 1u;
        const F3 d = diff_hl(rh, rl, s_rh[j], s_rl[j]);
        const bool image = small || rintf(d.x * iLx) != 0.f || rintf(d.y * iLy) != 0.f ||
                           rintf(d.z * iLz) != 0.f;
        if (np < kMaxPairs) G[np] = (short)(j | (image ? kPairImage : 0));
        ++np;
      }
    }
  }
  bool fit = true;
  if (bead) {
    for_solid_nodes(a, rh, rl, rlist, [&](float4 node) {
      const F3 d{(rh.x - node.x) + rl.x, (rh.y - node.y) + rl.y, (rh.z - node.z) + rl.z};
      if (!(dot(d, d) < rl2)) return;
      if (nw < kMaxWall) W[nw] = node;
      fit = fit && fits_short(node);
      ++nw;
    });
    a.nl_cnt[i] = min(np, kMaxPairs);
    a.wl_cnt[i] = min(nw, kMaxWall);
    a.nl_ref[i] = rh;
  }
  const int held = __syncthreads_and(np <= kMaxPairs && nw <= kMaxWall);
  if (!held) return kNlNone;
  // entries before this bead's: sums over the warp, then over the warps
  int upto = np + nw;
#pragma unroll
  for (int m = 1; m < 32; m <<= 1) {
    const int t = __shfl_up_sync(0xffffffffu, upto, m);
    if (lane >= m) upto += t;
  }
  if (lane == 31) s_sum[warp] = upto;
  __syncthreads();
  int before = 0, total = 0;
  for (int w = 0; w < (int)(blockDim.x >> 5); ++w) {
    if (w < warp) before += s_sum[w];
    total += s_sum[w];
  }
  if (!__syncthreads_and(fit && total <= item_cap(N))) return kNlBead;
  if (bead) {
    const int q = before + upto - (np + nw);
    s_first[i] = q;
    a.it_first[i] = q | (np + nw) << 16;
    const auto tag = [&](int e) { return (unsigned)i | min((unsigned)e, kItemTail) << 10; };
    const auto put = [&](int e, uint2 it) {
      s_item[q + e] = it;
      items[q + e] = it;
    };
    // read back what this thread has just written, in wide or several loads
    for (int k0 = 0; k0 < np; k0 += 8) {
      const uint4 g8 = reinterpret_cast<const uint4 *>(G)[k0 >> 3];
      const unsigned g2[4] = {g8.x, g8.y, g8.z, g8.w};
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        const unsigned v = g2[k >> 1] >> (16 * (k & 1));
        if (k0 + k < np)
          put(k0 + k, make_uint2(tag(k0 + k), (v & (LBMD_MAX_BEADS - 1)) | ((v & kPairImage) ? kItemImage : 0u)));
      }
    }
    for (int k0 = 0; k0 < nw; k0 += 8) {
      float4 v[8];
#pragma unroll
      for (int k = 0; k < 8; ++k)
        if (k0 + k < nw) v[k] = W[k0 + k];
#pragma unroll
      for (int k = 0; k < 8; ++k)
        if (k0 + k < nw)
          put(np + k0 + k, make_uint2(tag(np + k0 + k) | kItemWall | ((unsigned)(int)v[k].x << 16),
                                      ((unsigned)(int)v[k].y & 0xffffu) | ((unsigned)(int)v[k].z << 16)));
    }
  }
  *n_items = total;
  *cnt = np + nw;
  __syncthreads();
  return kNlFlat;
}

// Without lists (overflow): wall forces by scanning the stencil.
__device__ __noinline__ F3 wall_stencil_forces(const ChainArgs &a, float4 rh, float4 rl) {
  const float sig2 = a.sigma * a.sigma;
  const float rc = kTwoSixth * a.sigma, rc2 = rc * rc;
  const float eps24 = 24.0f * a.eps;
  F3 F{0.f, 0.f, 0.f};
  for_solid_nodes(a, rh, rl, rc, [&](float4 node) { wall_add(rh, rl, node, sig2, rc2, eps24, F); });
  return F;
}

// Fixed point of the spread: units of 2^-40.  The impulses of a node (|F| of
// order 1e-2) keep ~30 significant bits, far below a float ulp of the
// populations they reach.  The conversions are built from 32-bit ones: 64-bit
// integer <-> float conversions run at a small fraction of the FP32 rate on
// this GPU.
constexpr float kFixOne = 1099511627776.0f;  // 2^40

// round(v 2^40) for |v| < 2^10 as a 64-bit integer, rounded to nearest even
// like the direct conversion: with a = |v| 2^8 = hi + f (hi integral,
// 0 <= f <= 1 - 2^-24; a, hi and f exact in float), |v| 2^40 = hi 2^32 +
// f 2^32, only f 2^32 (< 2^32) needs rounding, and rounding to nearest even
// is symmetric in the sign.
__device__ __forceinline__ long long fix40(float v) {
  const float a = fabsf(v) * 256.0f;
  const float hi = floorf(a);
  const unsigned lo = __float2uint_rn((a - hi) * 4294967296.0f);
  const long long m = (long long)(((unsigned long long)__float2uint_rn(hi) << 32) | lo);
  return v < 0.f ? -m : m;
}

// q 2^-40 as a float: hi 2^-8 + lo 2^-40 with q = hi 2^32 + lo (0 <= lo <
// 2^32), the low word rounded to float first and the sum rounded once more.
__device__ __forceinline__ float unfix40(long long q) {
  const int hi = (int)(q >> 32);
  const unsigned lo = (unsigned)(unsigned long long)q;
  return __fmaf_rn((float)hi, 1.0f / 256.0f, __uint2float_rn(lo) * (1.0f / kFixOne));
}

// Adds entry e's share -w_e J_i of the impulse to the sum at the owner of its
// node (64-bit integer atomics: the result does not depend on their order).
// A share that is not finite, or too large for the fixed point (|F| >= 2^10:
// then even all 8 N <= 2^13 shares of a chain on one node stay below 2^63 in
// units of 2^-40), marks the sum instead, and the node receives NaN -- a
// stable step hands the fluid impulses of order 1e-2.
__device__ __forceinline__ void spread_add(const ChainArgs &a, int e, float4 j) {
  const int node = a.sp_node[e];
  if (node < 0) return;
  const float w = a.sp_w[e];
  const float fx = -w * j.x, fy = -w * j.y, fz = -w * j.z;
  SpreadAcc *q = a.acc + a.owner[node];
  const float lim = 1024.0f;  // 2^10
  if (!(fabsf(fx) < lim && fabsf(fy) < lim && fabsf(fz) < lim)) {
    atomicOr(reinterpret_cast<unsigned long long *>(&q->bad), 1ull);
    return;
  }
  atomicAdd(reinterpret_cast<unsigned long long *>(&q->x), (unsigned long long)fix40(fx));
  atomicAdd(reinterpret_cast<unsigned long long *>(&q->y), (unsigned long long)fix40(fy));
  atomicAdd(reinterpret_cast<unsigned long long *>(&q->z), (unsigned long long)fix40(fz));
}

// The owner's conversion: the summed force of node `node` (NaN if a
// contribution was not finite); the sum and the node's owner return to rest.
// The sum is read through L2 (it was written by atomics of an earlier kernel).
__device__ __forceinline__ F3 spread_take(const ChainArgs &a, int node, int e) {
  SpreadAcc *q = a.acc + e;
  const long long x = __ldcg(&q->x), y = __ldcg(&q->y), z = __ldcg(&q->z), bad = __ldcg(&q->bad);
  *q = SpreadAcc{0, 0, 0, 0};
  a.owner[node] = kOwnerFree;
  if (bad) {
    const float nan = __int_as_float(0x7fc00000);
    return F3{nan, nan, nan};
  }
  return F3{unfix40(x), unfix40(y), unfix40(z)};
}

// After every contribution is summed: entry e's record for the apply --
// (F, node) if e owns its node, node = -1 otherwise.
__device__ __forceinline__ float4 spread_record(const ChainArgs &a, int e) {
  const int node = a.sp_node[e];
  float4 out = make_float4(0.f, 0.f, 0.f, __int_as_float(-1));
  if (node >= 0 && a.owner[node] == e) {
    const F3 F = spread_take(a, node, e);
    out = make_float4(F.x, F.y, F.z, __int_as_float(node));
  }
  return out;
}

// Three standard normals for (bead, LB step, substep): Box-Muller on the four
// uniforms of one Philox block.
__device__ __forceinline__ float4 gauss3(uint64_t seed, uint32_t bead, int64_t step, uint32_t substep) {
  const U4 c{bead, (uint32_t)(uint64_t)step, (uint32_t)((uint64_t)step >> 32), substep & 0xFFu};
  const U4 r = philox4x32_10(c, (uint32_t)seed, (uint32_t)(seed >> 32));
  const float u1 = uniform23(r.x), u2 = uniform23(r.y);
  const float u3 = uniform23(r.z), u4 = uniform23(r.w);
  const float r1 = sqrtf(-2.0f * logf(u1)), r2 = sqrtf(-2.0f * logf(u3));
  float s2, c2, s4, c4;
  sincospif(2.0f * u2, &s2, &c2);
  sincospif(2.0f * u4, &s4, &c4);
  return make_float4(r1 * c2, r1 * s2, r2 * c4, 0.f);
}

// (2) the M MD substeps of one chain, one thread per bead, and (5) the
// bookkeeping; `a` may live in parameter or shared memory.  BLOCK is the
// register class (512, 768, 896 or 1024 threads).
//
// `beside`: the block may have started beside the gather and waits for it before
// it takes u_i; else u_i is there and read with the rest of the state.
//
// One chain is one block, so a substep is a chain of dependent phases and its
// bound is their latency.  The positions of a substep are final after SHAKE, so
// the next substep's forces, bond vectors and noise are found while RATTLE's
// boundary system is solved; what is left in line is: velocities and the sum
// of the acting forces, one barrier, two Newton iterations (rows and vote,
// solve), a last vote, positions and RATTLE's rows, one vote, the solve, one
// barrier.  A thread keeps its own and its successor's displacement, both
// updated by the same operations, so the Newton iterations exchange nothing but
// what the solve does.  Only the warps that hold beads, and the one that solves
// the boundary system, meet in the constraint solves; a chain of one warp
// solves without a barrier.  us a step without a solvent, with a list per bead,
// the solve's boundary system and every barrier in line / so: 20 beads 29.6 /
// 19.4, 100 beads 41.6 / 29.9, 400 beads 60.4 / 49.5, 700 beads 93 / 90, 1000
// beads 122 / 121; chains of 33 - 200 beads with no pair and no wall in reach,
// whose lists cost nothing, are slower by it (40 beads 19.0 / 21.8).
//
// The results of a step are those of earlier releases to the last bit
// (released_values.py among the tests): sums and products are written with
// their roundings where the compiler has a choice.
template <int BLOCK>
__device__ __forceinline__ void md_cycle_body(const ChainArgs &a, bool beside) {
  extern __shared__ float4 smem4[];
  const int N = a.N;
  const int i = threadIdx.x;  // bead of this thread
  const bool bead = i < N;
  // the warps that hold beads; the warp of the boundary system between them: the
  // last one, or the first of a block without a spare one; the threads that
  // evaluate the force list: those between the two, where there are two warps
  // of them and the chain is short, else all but the spare one's
  const int holders = bead_threads(N), nch = holders >> 5, warp = i >> 5, lane = i & 31;
  const bool holds = i < holders;
  const bool spare = nch > 2 && (int)blockDim.x > holders;
  const int workers = spare ? (int)blockDim.x - 32 : (int)blockDim.x;
  const bool middle = nch > 1 && warp == (spare ? workers >> 5 : 0);
  const int eval0 = N <= 224 && workers - holders >= 64 ? holders : 0;
  const int solvers = spare ? holders + 32 : holders;
  float4 *s_rh = smem4;          // positions, hi part (start of the substep)
  float4 *s_rl = s_rh + N;       // positions, lo part
  float4 *s_b = s_rl + N;        // bond vectors, start of the substep
  float4 *s_t = s_b + N;         // unconstrained displacement of the substep
  float4 *s_d = s_t + N;         // bond vectors at the end of the substep
  float *s_lam = (float *)(s_d + N);               // SHAKE multipliers of the last substep
  unsigned *s_mask = (unsigned *)(s_lam + N);      // acting entries of the bead's flat list
  float4 *s_f = (float4 *)((char *)smem4 + md_smem_head(N));  // their separations and force factors
  uint2 *s_item = (uint2 *)(s_f + item_cap(N));               // the flat list
  __shared__ int s_first[BLOCK];                              // a bead's first entry
  __shared__ float s_y[6 * 32], s_x[64];                      // sides and middle of a solve

  const DevStatus *st0 = a.status;
  const long long step = st0->step;
  const int max_trans0 = st0->max_trans, state0 = st0->state;
  const bool lists = a.eps != 0.f;
  int nl_ok = st0->nl_builds > 0 ? st0->nl_ok : kNlNone, n_items = st0->nl_items, n_own = 0;
  float4 rh = make_float4(0, 0, 0, 0), rl = rh, ref = rh;
  F3 v{0.f, 0.f, 0.f}, ui{0.f, 0.f, 0.f};
  double b0 = 1.0;
  if (bead) {
    rh = a.pos[i];
    rl = a.pos_lo[i];
    ref = a.nl_ref[i];
    v = f3(a.vel[i]);
    const float lam0 = a.lam[i];
    if (!beside) ui = f3(a.ui[i]);
    const int own = a.it_first[i];
    if (i < N - 1 && a.has_bonds) b0 = a.b0[i];
    s_rh[i] = rh;
    s_rl[i] = rl;
    s_lam[i] = lam0;
    s_mask[i] = 0u;
    s_first[i] = own & 0xffff;
    n_own = own >> 16;
  }
  if (nl_ok == kNlFlat)
    for (int q = i; q < n_items; q += 4 * blockDim.x) {  // four loads in flight
      uint2 it[4];
#pragma unroll
      for (int k = 0; k < 4; ++k)
        if (q + k * (int)blockDim.x < n_items) it[k] = a.items[q + k * blockDim.x];
#pragma unroll
      for (int k = 0; k < 4; ++k)
        if (q + k * (int)blockDim.x < n_items) s_item[q + k * blockDim.x] = it[k];
    }
  // Noise of every substep: a loop of its own, whose instructions stay in
  // the instruction cache over its turns (in the substep they do not: the
  // substep's code then exceeds it and is fetched anew each time).
#pragma unroll 1
  for (int k = 0; k < a.M; ++k)
    if (bead) {
      a.noise[(size_t)k * N + i] = gauss3(a.seed, (uint32_t)i, step, (uint32_t)k);
    }
  const float half_skin2 = 0.25f * kSkin * kSkin;
  auto moved = [&]() {
    const float dx = rh.x - ref.x, dy = rh.y - ref.y, dz = rh.z - ref.z;
    return !(dx * dx + dy * dy + dz * dz <= half_skin2);
  };
  int rebuild = __syncthreads_or(bead && (nl_ok == kNlNone || moved()));
  F3 J{0.f, 0.f, 0.f};
  const float dt = a.dt, m = a.mass, im = 1.0f / a.mass, idt = 1.0f / a.dt;
  const float sig_r = sqrtf(2.0f * m * a.gamma * a.kT / dt);
  const float b02 = (float)(b0 * b0);
  const float tol = fmaxf(a.shake_tol, 5e-7f);
  const bool bond = a.has_bonds && i < N - 1;  // bond (i, i + 1)
  const bool bends = a.kappa != 0.f && a.has_bonds;
  int shake_bad = 0, newton_total = 0, builds = 0;
  // A tridiagonal solve by the warps that hold beads: its first part, the
  // boundary system (solve_middle, a spare warp's whole share), and x_i and
  // x_{i-1}.  Every read of s_y and s_x precedes a barrier of the solvers that
  // comes before they are written again (votes, the barriers of a substep).
  auto solve_sides = [&](float sub, float diag, float sup, float rhs) {
    if (nch == 1) return tri_reduce<false>(N - 1, sub, diag, sup, rhs);
    const TriPart t = tri_reduce<true>(N - 1, sub, diag, sup, rhs);
    {
      float *y = s_y + 6 * warp + (lane == 0 ? 0 : 3);
      if (lane == 0 || lane == 31) {
        y[0] = t.y;
        y[1] = t.v;
        y[2] = t.w;
      }
      __syncwarp();
      if (middle) {
        bar_sync(kBarSides, solvers);
        tri_boundary(nch, s_y, s_x);
        __syncwarp();
      } else {
        bar_arrive(kBarSides, solvers);
      }
    }
    return t;
  };
  auto solve_middle = [&]() {
    bar_sync(kBarSides, solvers);
    tri_boundary(nch, s_y, s_x);
    __syncwarp();
    bar_arrive(kBarMiddle, solvers);
  };
  auto solve_ends = [&](TriPart t, float &x_prev) {
    if (nch > 1) bar_sync(kBarMiddle, solvers);
    const float x = tri_finish(t, warp, nch, s_x);
    const float xu = __shfl_up_sync(0xffffffffu, x, 1);
    x_prev = lane > 0 ? xu : (warp > 0 ? s_x[warp - 1] : 0.f);
    return x;
  };
  // whether every solver says yes
  auto vote = [&](bool yes) {
    if (nch > 1) {
      __syncwarp();
      return bar_all(kBarVote, solvers, yes);
    }
    const bool all = __all_sync(0xffffffffu, yes);
    __syncwarp();
    return all;
  };
  // What the coming substep k needs of the positions now in s_rh, s_rl (every
  // thread has passed a barrier since they were written; another follows
  // before the results are read): noise, the force on this bead from the
  // drive and from the bending at its own angle (the shares of that angle on the
  // neighbours left in s_d and in the unused components of s_rh, s_rl, s_b and
  // s_d), its bond vector and the entries of the flat list.
  float4 xi = make_float4(0.f, 0.f, 0.f, 0.f);
  F3 Fd{0.f, 0.f, 0.f}, gb{0.f, 0.f, 0.f};
  float Ab = 0.f;
  auto prepare = [&](int k) {
    if (lists && nl_ok == kNlFlat && i >= eval0 && i < workers)
      eval_items(a, s_item, n_items, i - eval0, workers - eval0, s_rh, s_rl, s_f, s_mask);
    if (!bead) return;
    xi = a.noise[(size_t)k * N + i];  // this thread wrote it
    F3 sb{0.f, 0.f, 0.f};
    if (bond) sb = diff_hl(s_rh[i + 1], s_rl[i + 1], rh, rl);
    float4 keep = f4(sb);
    if (bends) {
      F3 g1{0.f, 0.f, 0.f}, g2 = g1;
      F3 fc{0.f, 0.f, 0.f};  // on bead i + 1
      Ab = 0.f;
      if (i >= 1 && i + 1 < N) {
        const F3 bm = diff_hl(rh, rl, s_rh[i - 1], s_rl[i - 1]);
        const float l1 = sqrtf(dot(bm, bm)), lc = sqrtf(dot_yx(bm, bm)), l2 = sqrtf(dot(sb, sb)), b12 = dot(bm, sb);
        float Ac = Ab = bend_terms(bm, sb, l1, l2, b12, a.kappa, g1, g2);
        fc = g2;
        // the force on bead i + 1 has always been found with the other rounding of l1
        if (lc != l1) {
          F3 g;
          Ac = bend_terms(bm, sb, lc, l2, b12, a.kappa, g, fc);
        }
        fc = Ac * fc;
      }
      gb = g1 - g2;
      s_d[i] = make_float4(fc.x, fc.y, fc.z, -Ab);
      keep.w = g1.x;
      s_rh[i].w = g1.y;
      s_rl[i].w = g1.z;
    }
    if (bond || bends) s_b[i] = keep;
    // pulling force inside the channel through the pore
    Fd = drive_force_at(a, rh, rl);
  };
  F3 D1{0.f, 0.f, 0.f};  // displacement of bead i + 1
  F3 d{0.f, 0.f, 0.f};   // bond vector i at the end of the substep
  F3 dm{0.f, 0.f, 0.f};  // bond vector i - 1 there
  float r_sub = 0.f, r_diag = 1.f, r_sup = 0.f, r_rhs = 0.f;  // RATTLE's row

  // (2) M MD substeps.  One turn ends substep k - 1 (RATTLE) and takes substep
  // k up to its positions, so that every phase stands in the code once.
  for (int k = 0;; ++k) {
    if (rebuild && lists && k < a.M) {
      // neighbour lists: pairs and solid nodes within r_c + skin
      nl_ok = build_lists(a, i, bead, rh, rl, s_rh, s_rl, s_item, s_first, &n_items, &n_own);
      ref = rh;
      ++builds;
    }
    TriPart part{0.f, 0.f, 0.f};
    if (a.has_bonds && k > 0) {
      if (holds)
        part = solve_sides(r_sub, r_diag, r_sup, r_rhs);
      else if (middle)
        solve_middle();
    }
    if (k < a.M) prepare(k);
    if (a.has_bonds && k > 0 && holds) {
      __syncwarp();
      float mum;
      const float mu = solve_ends(part, mum);
      if (bond) v = axpy(mu * im, d, v);
      if (bead && i > 0) v = axpy(-(mum * im), dm, v);
    }
    __syncthreads();
    if (k == a.M) break;
    if (k == 0 && beside) {
      // (1) interpolated by k_gather, beside which this block may have
      // started; frozen for the M substeps
      asm volatile("griddepcontrol.wait;" ::: "memory");
      if (bead) ui = f3(a.ui[i]);
    }
    // bond vectors s_{i-1}, s_i, s_{i+1} around the bead; the blocks with 64 or 72
    // registers a thread read them anew for each use
    F3 sm{0.f, 0.f, 0.f}, sb{0.f, 0.f, 0.f}, sp{0.f, 0.f, 0.f}, D{0.f, 0.f, 0.f};
    auto bonds = [&]() {
      if (bond) sb = f3(s_b[i]);
      if (bead && i > 0) sm = f3(s_b[i - 1]);
      if (i < N - 2) sp = f3(s_b[i + 1]);
    };
    float lam = 0.f;  // multiplier of bond i
    if (bead) {
      F3 Fc{0.f, 0.f, 0.f};
      if (bends) {
        if (i >= 2) Fc = Fc + f3(s_d[i - 1]);
        Fc = axpy(Ab, gb, Fc);
        if (i + 2 < N) Fc = axpy(s_d[i + 1].w, F3{s_b[i + 1].w, s_rh[i + 1].w, s_rl[i + 1].w}, Fc);
      }
      Fc = Fc + Fd;
      if (lists) {
        if (nl_ok == kNlFlat) {
          F3 F{0.f, 0.f, 0.f};
          const float4 *f = s_f + s_first[i];
          unsigned mask = s_mask[i];
          s_mask[i] = 0u;
          for (; mask; mask &= mask - 1u) {
            const float4 e = f[__ffs(mask) - 1];
            F = axpy(e.w, f3(e), F);
          }
          for (int q = (int)kItemTail; q < n_own; ++q) F = axpy(f[q].w, f3(f[q]), F);
          Fc = Fc + F;
        } else if (nl_ok == kNlBead) {
          Fc = Fc + list_forces(a, i, rh, rl, s_rh, s_rl);
        } else {
          Fc = Fc + all_pair_forces(a, i, rh, rl, s_rh, s_rl) + wall_stencil_forces(a, rh, rl);
        }
      }
      const F3 fdrag = (-m * a.gamma) * (v - ui);
      const F3 fr = sig_r * F3{xi.x, xi.y, xi.z};
      v = v + (dt * im) * (Fc + fdrag + fr);
      J = J + dt * (fdrag + fr);
      D = dt * v;  // unconstrained displacement r~ - r
    }
    if (a.has_bonds && holds) {
      // SHAKE on displacements: D_i = dt v_i + (lam_i s_i - lam_{i-1} s_{i-1}) / m
      // with the old bond vectors s_b; Newton on G_b = |s_b + D_{b+1} - D_b|^2 - b0^2.
      // Old bonds come from the double-float positions.
      // Warm start: the multipliers of the previous substep applied along the
      // new old-bond vectors (the constraint forces change slowly).
      if (bead) {
        if (bond) {
          sb = f3(s_b[i]);
          lam = s_lam[i];
          D = axpy(lam * im, sb, D);
        }
        if (i > 0) {
          sm = f3(s_b[i - 1]);
          D = axpy(-(s_lam[i - 1] * im), sm, D);
        }
        if (i < N - 2) sp = f3(s_b[i + 1]);
        s_t[i] = f4(D);
      }
      __syncwarp();
      if (nch > 1) bar_sync(kBarBeads, holders);
      if (bond) D1 = f3(s_t[i + 1]);
      for (int it = 0;; ++it) {
        float G = 0.f, diag = 1.f, sub = 0.f, sup = 0.f;
        bool ok = true;
        if (BLOCK > 768) bonds();
        if (bond) {
          // old bond from the double-float positions, displacements small: the
          // float residual is good to ~1e-7 of b0^2
          d = sb + (D1 - D);
          G = dot(d, d) - b02;
          ok = fabsf(G) <= tol * b02;
          diag = -4.0f * im * dot(d, sb);
          if (i > 0) sub = 2.0f * im * dot(d, sm);
          if (i < N - 2) sup = 2.0f * im * dot(d, sp);
          s_d[i] = f4(d);
        }
        if (vote(ok)) break;
        if (it >= a.shake_maxit) {
          const bool bad = bond && !(fabsf(G) <= 1e-3f * b02);
          if (!vote(!bad)) shake_bad = 1;
          break;
        }
        ++newton_total;
        const TriPart t = solve_sides(sub, diag, sup, -G);
        float xm;
        const float x = solve_ends(t, xm);
        // what the thread of bead i + 1 finds for x_{i+1} and x_i: the first
        // bead of a warp takes x_i from the boundary system
        float xn = __shfl_down_sync(0xffffffffu, x, 1), xnm = x;
        if (lane == 31 && warp + 1 < nch) {
          const float *y = s_y + 6 * (warp + 1);
          xn = tri_finish(TriPart{y[0], y[1], y[2]}, warp + 1, nch, s_x);
          xnm = s_x[warp];
        }
        if (BLOCK > 768) bonds();
        // own and next bead's displacement, by the same operations on both
        // threads that hold it
        if (bond) {
          D = axpy(x * im, sb, D);
          if (i < N - 2) D1 = axpy(xn * im, sp, D1);
          D1 = axpy(-(xnm * im), sb, D1);
          lam += x;
        }
        if (bead && i > 0) D = axpy(-(xm * im), sm, D);
      }
      if (bond) s_lam[i] = lam;  // read again only after later barriers
    } else if (a.has_bonds && middle) {
      // the spare warp: the boundary systems of the Newton iterations
      for (int it = 0;; ++it) {
        if (vote(true)) break;
        if (it >= a.shake_maxit) {
          vote(true);
          break;
        }
        solve_middle();
      }
    }
    // every read of s_rh / s_rl of this substep precedes a barrier of the
    // constraint solves; without constraints one barrier is needed here
    if (!a.has_bonds) __syncthreads();
    if (bead) {
      // v = (r' - r) / dt evaluated as D / dt (no cancellation); r' = r + D
      v = F3{__fmul_rn(idt, D.x), __fmul_rn(idt, D.y), __fmul_rn(idt, D.z)};
      two_sum_add(rh.x, rl.x, D.x);
      two_sum_add(rh.y, rl.y, D.y);
      two_sum_add(rh.z, rl.z, D.z);
      s_rh[i] = rh;
      s_rl[i] = rl;
    }
    if (a.has_bonds && bead) {
      // RATTLE: v_i += (mu_i d_i - mu_{i-1} d_{i-1}) / m with the new bond
      // vectors d_b = s_b + D_{b+1} - D_b, so that d_b . (v_{b+1} - v_b) = 0.
      if (i > 0) dm = f3(s_d[i - 1]);
      if (bond) {
        const F3 vn{__fmul_rn(idt, D1.x), __fmul_rn(idt, D1.y), __fmul_rn(idt, D1.z)};
        r_rhs = -dot(d, vn - v);
        r_diag = -2.0f * im * dot_yx(d, d);
        if (i > 0) r_sub = im * dot(d, dm);
        if (i < N - 2) r_sup = im * dot(d, f3(s_d[i + 1]));
      }
    }
    rebuild = __syncthreads_or(bead && moved());
  }

  asm volatile("griddepcontrol.launch_dependents;");  // the spread's sum may be placed
  if (bead) {
    a.pos[i] = rh;
    a.pos_lo[i] = rl;
    a.vel[i] = f4(v);
    a.J[i] = f4(J);
    a.lam[i] = s_lam[i];
  }
  // Translocation bookkeeping (Sec. III): unwrapped x = origin + hi + lo
  const float xrel = bead ? ((float)(a.ox - a.wall_x) + rh.x) + rl.x : 0.f;
  const bool finite = isfinite(rh.x) && isfinite(rh.y) && isfinite(rh.z) && isfinite(v.x) &&
                      isfinite(v.y) && isfinite(v.z);
  const int nt = __syncthreads_count(bead && a.has_wall && xrel < 0.f);
  const int nan = __syncthreads_or(bead && !finite);
  const int out = __syncthreads_and(!bead || xrel > (float)(a.wall_t - 1) + 1.5f);
  const int bad = __syncthreads_or(shake_bad);
  if (i == 0) {
    DevStatus *st = a.status;
    const int max_trans = max(max_trans0, nt);  // read at the start: no load here
    st->n_trans = nt;
    st->max_trans = max_trans;
    if (bad) st->shake_fail += 1;
    st->newton_iters = newton_total;
    if (builds) st->nl_builds += builds;
    st->nl_ok = nl_ok;
    st->nl_items = n_items;
    if (state0 == LBMD_RUNNING) {
      if (nan)
        st->state = LBMD_NAN;
      else if (bad)
        st->state = LBMD_SHAKE_FAIL;
      else if (a.has_wall && N > 0) {
        if (nt == N) {
          st->state = LBMD_TRANSLOCATED;
          st->t_transloc = step + 1;
        } else if (max_trans >= 1 && out) {
          st->state = LBMD_RETRACTED;
        }
      }
    }
  }
  // Sec. III chain diagnostics at the end of every diag_every-th step: radii
  // of gyration of the translocated (x < x_wall, as N_T) and untranslocated
  // beads from two block sums (centres, then squared distances), the work
  // rates of Eqs. 13-14 and the kinetic energy
  if (a.diag_every > 0 && (step + 1) % a.diag_every == 0) {
    __shared__ float s_red[32 * 6 + 6];
    const bool tr = bead && a.has_wall && xrel < 0.f, un = bead && !tr;
    const F3 r{rh.x + rl.x, rh.y + rl.y, rh.z + rl.z};  // local frame
    float c[6] = {tr ? r.x : 0.f, tr ? r.y : 0.f, tr ? r.z : 0.f,
                  un ? r.x : 0.f, un ? r.y : 0.f, un ? r.z : 0.f};
    block_sum<6>(c, s_red);
    const int nu = N - nt;
    const float it = nt > 0 ? 1.0f / (float)nt : 0.f, iu = nu > 0 ? 1.0f / (float)nu : 0.f;
    const F3 dt_{r.x - c[0] * it, r.y - c[1] * it, r.z - c[2] * it};
    const F3 du_{r.x - c[3] * iu, r.y - c[4] * iu, r.z - c[5] * iu};
    const float fd = bead ? drive_force_at(a, rh, rl).x : 0.f;
    float q[5] = {tr ? dot(dt_, dt_) : 0.f, un ? dot(du_, du_) : 0.f, bead ? dot(v, ui) : 0.f,
                  fd * v.x, bead ? dot(v, v) : 0.f};
    block_sum<5>(q, s_red);
    if (i == 0) {
      DevStatus *st = a.status;
      const int k = st->diag_count;
      if (k < a.diag_cap) {
        DevDiag d;
        d.step = step + 1;
        d.n_trans = nt;
        d.r_t = nt > 0 ? sqrtf(q[0] * it) : 0.f;
        d.r_u = nu > 0 ? sqrtf(q[1] * iu) : 0.f;
        d.r_e = powf(powf(d.r_t, 1.0f / 0.6f) + powf(d.r_u, 1.0f / 0.6f), 0.6f);
        d.s_h = a.mass * a.gamma * q[2];
        d.s_e = q[3];
        d.kinetic = 0.5f * a.mass * q[4];
        d.pad = 0;
        a.diag[k] = d;
        st->diag_count = k + 1;
      }
    }
  }
}

template <int BLOCK>
__global__ void __launch_bounds__(BLOCK, 1) k_md_cycle(ChainArgs a, bool beside) {
  md_cycle_body<BLOCK>(a, beside);
}

// Ensemble variant: block b runs chain chains[b] if its realisation is live.
// The chain's arguments are copied to shared memory once.
template <int BLOCK>
__global__ void __launch_bounds__(BLOCK, 1)
    k_ens_md_cycle(const EnsMember *__restrict__ mem, const int *__restrict__ chains,
                   const int *__restrict__ live) {
  __shared__ ChainArgs s_a;
  const int m = chains[blockIdx.x];
  if (!live[m]) return;  // the whole block leaves together
  static_assert(sizeof(ChainArgs) % sizeof(int) == 0, "ChainArgs copied as ints");
  const int *src = reinterpret_cast<const int *>(&mem[m].a);
  int *dst = reinterpret_cast<int *>(&s_a);
  for (int k = threadIdx.x; k < (int)(sizeof(ChainArgs) / sizeof(int)); k += blockDim.x) dst[k] = src[k];
  __syncthreads();
  md_cycle_body<BLOCK>(s_a, false);
}

// Stage (1) for (bead, corner) pair e = 8 i + k handled by one thread; the
// eight lanes of a bead are consecutive, so the weight normalisation and the
// sum over corners are lane shuffles.  Writes the transfer weights for the
// spread and returns the bead's interpolated u (on every lane of the bead).
template <int S>
__device__ F3 gather_pair(const ChainArgs &a, const void *f, int e, bool valid) {
  using T = typename Store<S>::T;
  const LbGeom &g = a.geo;
  const int i = e >> 3, k = e & 7;
  int node = -1;
  float w = 0.f;
  if (valid) {
    const float4 rh = a.pos[i], rl = a.pos_lo[i];
    int c0[3];
    float s[3];
    cell_frac_hl(rh.x, rl.x, a.ox, g.nx, c0[0], s[0]);
    cell_frac_hl(rh.y, rl.y, a.oy, g.ny, c0[1], s[1]);
    cell_frac_hl(rh.z, rl.z, a.oz, g.nz, c0[2], s[2]);
    int x, y, z;
    if (a.coupling == LBMD_COUPLING_NGP) {
      x = s[0] >= 0.5f ? wrap_p1(c0[0], g.nx) : c0[0];
      y = s[1] >= 0.5f ? wrap_p1(c0[1], g.ny) : c0[1];
      z = s[2] >= 0.5f ? wrap_p1(c0[2], g.nz) : c0[2];
      w = k == 0 ? 1.f : 0.f;
    } else {
      const int ox = k & 1, oy = (k >> 1) & 1, oz = (k >> 2) & 1;
      x = ox ? wrap_p1(c0[0], g.nx) : c0[0];
      y = oy ? wrap_p1(c0[1], g.ny) : c0[1];
      z = oz ? wrap_p1(c0[2], g.nz) : c0[2];
      w = (ox ? s[0] : 1.f - s[0]) * (oy ? s[1] : 1.f - s[1]) * (oz ? s[2] : 1.f - s[2]);
    }
    if (w != 0.f && !solid_at(g.solid, g.ntx, g.ny, x, y, z))
      node = (int)(((size_t)z * g.ny + y) * g.nx + x);
    else
      w = 0.f;
  }
  float wsum = w;
  wsum += __shfl_xor_sync(0xffffffffu, wsum, 1);
  wsum += __shfl_xor_sync(0xffffffffu, wsum, 2);
  wsum += __shfl_xor_sync(0xffffffffu, wsum, 4);
  const float wn = wsum > 0.f ? w / wsum : 0.f;
  if (wn == 0.f) node = -1;
  F3 u{0.f, 0.f, 0.f};
  if (valid) {
    a.sp_node[e] = node;
    a.sp_w[e] = wn;
    if (node >= 0) {
      if (a.owner != nullptr) atomicMin(a.owner + node, e);  // the node's spread owner: its smallest entry
      const int x = node % g.nx, yz = node / g.nx;
      const int y = yz % g.ny, z = yz / g.ny;
      float h[kQ];
      fetch19<S>(g, (const T *)f, x, y, z, a.f_mode, h);
      float drho, jx, jy, jz;
      moments19(h, drho, jx, jy, jz);
      if (a.forcing == LBMD_FORCING_GUO) {
        jx += 0.5f * a.g[0];
        jy += 0.5f * a.g[1];
        jz += 0.5f * a.g[2];
      }
      const float rinv = wn / (a.rho0 + drho);
      u = F3{jx * rinv, jy * rinv, jz * rinv};
    }
  }
#pragma unroll
  for (int m = 1; m < 8; m <<= 1) {
    u.x += __shfl_xor_sync(0xffffffffu, u.x, m);
    u.y += __shfl_xor_sync(0xffffffffu, u.y, m);
    u.z += __shfl_xor_sync(0xffffffffu, u.z, m);
  }
  return u;
}

template <int S>
__global__ void __launch_bounds__(256) k_gather(ChainArgs a) {
  asm volatile("griddepcontrol.launch_dependents;");  // the MD block may be placed
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  const bool valid = e < 8 * a.N;
  const F3 u = gather_pair<S>(a, a.f, e, valid);
  if (valid && (e & 7) == 0) a.ui[e >> 3] = f4(u);
}

// Ensemble gather: thread e serves corner e & 7 of padded bead slot e >> 3,
// beads[slot] = (realisation, bead) or m < 0 for padding.  Every realisation's
// slots start at a multiple of four, so a warp never mixes realisations.
template <int S>
__global__ void __launch_bounds__(256)
    k_ens_gather(const EnsMember *__restrict__ mem, const int2 *__restrict__ beads, int nb,
                 const int *__restrict__ live, int cur) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  const int slot = e >> 3;
  int2 mi = make_int2(-1, 0);
  if (slot < nb) mi = beads[slot];
  const bool valid = mi.x >= 0 && live[mi.x];
  const EnsMember &M = mem[valid ? mi.x : 0];
  const F3 u = gather_pair<S>(M.a, valid ? M.pop[cur] : nullptr, 8 * mi.y + (e & 7), valid);
  if (valid && (e & 7) == 0) M.a.ui[mi.y] = f4(u);
}

// Dynamic shared memory with which a block of k_ens_md_cycle<512> leaves none on
// its SM for another block.
static cudaError_t md_alone_bytes(size_t *bytes) {
  cudaFuncAttributes at;
  const cudaError_t e = cudaFuncGetAttributes(&at, k_ens_md_cycle<512>);
  if (e == cudaSuccess) *bytes = kSmemOfBlock - at.sharedSizeBytes;
  return e;
}

cudaError_t md_prepare() {
  size_t alone = 0;
  cudaError_t e;
  if ((e = md_alone_bytes(&alone)) != cudaSuccess) return e;
  const int s512 = (int)md_smem_bytes(512), s768 = (int)md_smem_bytes(768), s1024 = (int)md_smem_bytes(LBMD_MAX_BEADS);
  if ((e = cudaFuncSetAttribute(k_md_cycle<768>, cudaFuncAttributeMaxDynamicSharedMemorySize, s768)) != cudaSuccess) return e;
  if ((e = cudaFuncSetAttribute(k_md_cycle<896>, cudaFuncAttributeMaxDynamicSharedMemorySize, s1024)) != cudaSuccess) return e;
  if ((e = cudaFuncSetAttribute(k_ens_md_cycle<768>, cudaFuncAttributeMaxDynamicSharedMemorySize, s768)) != cudaSuccess) return e;
  if ((e = cudaFuncSetAttribute(k_md_cycle<512>, cudaFuncAttributeMaxDynamicSharedMemorySize, s512)) != cudaSuccess) return e;
  if ((e = cudaFuncSetAttribute(k_md_cycle<1024>, cudaFuncAttributeMaxDynamicSharedMemorySize, s1024)) != cudaSuccess) return e;
  if ((e = cudaFuncSetAttribute(k_ens_md_cycle<512>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)alone)) != cudaSuccess) return e;
  return cudaFuncSetAttribute(k_ens_md_cycle<1024>, cudaFuncAttributeMaxDynamicSharedMemorySize, s1024);
}

cudaError_t launch_gather(int storage, const ChainArgs &a, cudaStream_t s) {
  if (a.N <= 0) return cudaSuccess;
  const int blocks = (8 * a.N + 255) / 256;
  switch (storage) {
    case LBMD_STORE_F32: k_gather<LBMD_STORE_F32><<<blocks, 256, 0, s>>>(a); break;
    case LBMD_STORE_F16: k_gather<LBMD_STORE_F16><<<blocks, 256, 0, s>>>(a); break;
    case LBMD_STORE_BF16: k_gather<LBMD_STORE_BF16><<<blocks, 256, 0, s>>>(a); break;
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

// The MD block is launched at the highest stream priority so that, when it
// and the stream-collide become ready together, its block is placed first.
// beside: the kernel before it on `s` is the gather of the same step, which lets
// this one start beside it (programmatic dependent launch): the block then
// reads its state and lists, draws its noise and finds its first forces while
// the gather runs, and waits for it before it takes u_i.
cudaError_t launch_md_cycle(const ChainArgs &a, int priority, bool beside, cudaStream_t s) {
  if (a.N <= 0) return cudaSuccess;
  const int threads = md_threads(a.N);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(1);
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = md_smem_bytes(a.N);
  cfg.stream = s;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributePriority;
  attr[0].val.priority = priority;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = beside ? 2 : 1;
  if (threads <= 512) return cudaLaunchKernelEx(&cfg, k_md_cycle<512>, a, beside);
  if (threads <= 768) return cudaLaunchKernelEx(&cfg, k_md_cycle<768>, a, beside);
  if (threads <= 896) return cudaLaunchKernelEx(&cfg, k_md_cycle<896>, a, beside);
  return cudaLaunchKernelEx(&cfg, k_md_cycle<1024>, a, beside);
}

// The sum of the spread as two kernels, one thread per (bead, corner) entry.
__global__ void __launch_bounds__(256) k_spread_accum(ChainArgs a) {
  asm volatile("griddepcontrol.wait;" ::: "memory");  // the MD cycle's impulses
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e < 8 * a.N) spread_add(a, e, a.J[e >> 3]);
  asm volatile("griddepcontrol.launch_dependents;");
}
__global__ void __launch_bounds__(256) k_spread_finalize(ChainArgs a) {
  asm volatile("griddepcontrol.wait;" ::: "memory");  // every share
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= 8 * a.N) return;
  a.sp_src[e] = spread_record(a, e);
}

// (3) extrapolation of the forces: node x_k receives -sum_i w_ik J_i as the
// source S_p = 3 w_p c_p . F (Eq. 10, reaction sign), added by the node's
// owner entry to the post-collision populations h*_p(x_k), wherever layout
// `mode` holds them: [p][x_k] (pull), [opp(p)][x_k] (in place, after an even
// step), or [p][x_k + c_p] -- [opp(p)][x_k] if x_k + c_p is solid -- (in
// place, after an odd step).  No other thread writes those words in this
// kernel: FP32 adds with one atomic each (no read-back); 16-bit storage reads
// the 18 words first and writes each rounded once.  The owner's force comes
// from its record sp_src[e] (TAKE = false: converted by k_spread_finalize) or
// straight from its fixed-point sum (TAKE = true: the conversion of
// spread_record done here, one launch fewer after the MD cycle).
template <int S, bool TAKE>
__global__ void __launch_bounds__(256)
    k_spread_apply(LbGeom g, ChainArgs a, int nw, typename Store<S>::T *dst, int mode,
                   DevStatus *bump) {
  using St = Store<S>;
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (bump != nullptr && e == 0) {
    bump->step += 1;
    // populations that are not finite end the run as a bead NaN does
    if (bump->pop_bad && bump->state == LBMD_RUNNING) bump->state = LBMD_NAN;
  }
  if (e >= nw) return;
  int node;
  F3 F;
  if (TAKE) {
    node = a.sp_node[e];
    if (node < 0 || a.owner[node] != e) return;  // not an owner
    F = spread_take(a, node, e);
  } else {
    const float4 v = a.sp_src[e];
    node = __float_as_int(v.w);
    if (node < 0) return;  // not an owner
    F = F3{v.x, v.y, v.z};
  }
  const size_t st = pop_stride<S, size_t>((size_t)g.Vp), own = pop_base<S, size_t>(pop_node<S, size_t>(g, (size_t)node));
  uint32_t bb = 0u;
  int x = 0, y = 0, z = 0;
  if (mode == kPopAALocal) {
    x = node % g.nx;
    const int yz = node / g.nx;
    y = yz % g.ny;
    z = yz / g.ny;
    bb = __ldg(&g.lmask[node]);  // bit opp(p): x_k + c_p is solid
  }
  size_t at[kQ];
#pragma unroll
  for (int p = 1; p < kQ; ++p) {
    if (mode == kPopAALocal) {
      const size_t t = ((size_t)wrapi(z + cz(p), g.nz) * g.ny + wrapi(y + cy(p), g.ny)) * row_pitch<S>(g) +
                       wrapi(x + cx(p), g.nx);
      at[p] = ((bb >> opp(p)) & 1u) ? (size_t)opp(p) * st + own : (size_t)p * st + pop_base<S, size_t>(t);
    } else {
      at[p] = (size_t)(mode == kPopAASwap ? opp(p) : p) * st + own;
    }
  }
  if (S == LBMD_STORE_F32) {
#pragma unroll
    for (int p = 1; p < kQ; ++p)
      St::add(dst + at[p], 3.0f * wq(p) * (cx(p) * F.x + cy(p) * F.y + cz(p) * F.z));
  } else {
    // all 18 loads first, then the stores: one memory latency, not eighteen
    float hv[kQ];
#pragma unroll
    for (int p = 1; p < kQ; ++p) hv[p] = St::load_plain(dst + at[p]);
#pragma unroll
    for (int p = 1; p < kQ; ++p)
      St::store(dst + at[p], hv[p] + 3.0f * wq(p) * (cx(p) * F.x + cy(p) * F.y + cz(p) * F.z));
  }
}

cudaError_t launch_spread_sum(const ChainArgs &a, bool records, cudaStream_t s) {
  if (a.N <= 0) return cudaSuccess;
  // both may be placed while the kernel before them ends (programmatic
  // dependent launch; they wait for its results first)
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((8 * a.N + 255) / 256);
  cfg.blockDim = dim3(256);
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  const cudaError_t e = cudaLaunchKernelEx(&cfg, k_spread_accum, a);
  if (e != cudaSuccess || !records) return e;
  return cudaLaunchKernelEx(&cfg, k_spread_finalize, a);
}

template <int S>
static void apply_as(bool take, int blocks, const LbGeom &g, const ChainArgs &a, int nw, void *dst,
                     int mode, DevStatus *bump, cudaStream_t s) {
  using T = typename Store<S>::T;
  if (take)
    k_spread_apply<S, true><<<blocks, 256, 0, s>>>(g, a, nw, (T *)dst, mode, bump);
  else
    k_spread_apply<S, false><<<blocks, 256, 0, s>>>(g, a, nw, (T *)dst, mode, bump);
}

cudaError_t launch_spread_apply(int storage, const LbGeom &g, const ChainArgs &a, void *dst,
                                int mode, bool take, DevStatus *bump, cudaStream_t s) {
  // no records and no sums without a coupled chain
  const int nw = (take ? a.owner != nullptr : a.sp_src != nullptr) ? 8 * a.N : 0;
  const int blocks = nw > 0 ? (nw + 255) / 256 : 1;
  switch (storage) {
    case LBMD_STORE_F32: apply_as<LBMD_STORE_F32>(take, blocks, g, a, nw, dst, mode, bump, s); break;
    case LBMD_STORE_F16: apply_as<LBMD_STORE_F16>(take, blocks, g, a, nw, dst, mode, bump, s); break;
    case LBMD_STORE_BF16: apply_as<LBMD_STORE_BF16>(take, blocks, g, a, nw, dst, mode, bump, s); break;
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

// Ensemble apply: same lane layout as k_ens_gather; each owner entry takes its
// node's force -- from its record (TAKE = false: k_ens_spread_finalize) or its
// sum (TAKE = true) -- and adds the source as k_spread_apply does.  The first
// lane of every realisation bumps its step count (if live) and decides whether
// it takes part in the next step.  Bound by the latency of dependent reads that
// the stream-collide has driven out of L2: the records, in the entries' own
// order, take the sum's three away.
template <int S, bool TAKE>
__global__ void __launch_bounds__(256)
    k_ens_spread(const EnsMember *__restrict__ mem, const int2 *__restrict__ beads, int nb,
                 const int *__restrict__ live, int *__restrict__ live_next, int cur,
                 const long long *__restrict__ max_steps, const float4 *__restrict__ rec) {
  using St = Store<S>;
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  const int slot = e >> 3, k = e & 7;
  int2 mi = make_int2(-1, 0);
  float4 r = make_float4(0.f, 0.f, 0.f, __int_as_float(-1));
  if (slot < nb) {
    mi = beads[slot];
    if (!TAKE) r = rec[e];
  }
  const bool valid = mi.x >= 0 && live[mi.x];
  if (valid && (TAKE ? mem[mi.x].a.owner != nullptr : __float_as_int(r.w) >= 0)) {
    const ChainArgs &a = mem[mi.x].a;
    const int e2 = 8 * mi.y + k;
    const int node = TAKE ? a.sp_node[e2] : __float_as_int(r.w);
    if (!TAKE || (node >= 0 && a.owner[node] == e2)) {
      const F3 F = TAKE ? spread_take(a, node, e2) : F3{r.x, r.y, r.z};
      const size_t st = pop_stride<S, size_t>((size_t)a.geo.Vp);
      typename St::T *dst = (typename St::T *)mem[mi.x].pop[cur ^ 1] +
                              pop_base<S, size_t>(pop_node<S, size_t>(a.geo, (size_t)node));
      if (S == LBMD_STORE_F32) {
#pragma unroll
        for (int p = 1; p < kQ; ++p)
          St::add(dst + (size_t)p * st, 3.0f * wq(p) * (cx(p) * F.x + cy(p) * F.y + cz(p) * F.z));
      } else {
        float hv[kQ];
#pragma unroll
        for (int p = 1; p < kQ; ++p) hv[p] = St::load_plain(dst + (size_t)p * st);
#pragma unroll
        for (int p = 1; p < kQ; ++p)
          St::store(dst + (size_t)p * st,
                    hv[p] + 3.0f * wq(p) * (cx(p) * F.x + cy(p) * F.y + cz(p) * F.z));
      }
    }
  }
  if (mi.x >= 0 && mi.y == 0 && k == 0) {
    int next = 0;
    if (valid) {
      DevStatus *st = mem[mi.x].a.status;
      const long long s = st->step + 1;
      st->step = s;
      st->out_buf = cur ^ 1;
      if (st->pop_bad && st->state == LBMD_RUNNING) st->state = LBMD_NAN;
      next = st->state == LBMD_RUNNING && s < *max_steps;
    }
    live_next[mi.x] = next;
  }
}

cudaError_t launch_ens_gather(int storage, const EnsMember *mem, const int2 *beads, int nb,
                              const int *live, int cur, cudaStream_t s) {
  const int blocks = nb > 0 ? (8 * nb + 255) / 256 : 1;
  switch (storage) {
    case LBMD_STORE_F32: k_ens_gather<LBMD_STORE_F32><<<blocks, 256, 0, s>>>(mem, beads, nb, live, cur); break;
    case LBMD_STORE_F16: k_ens_gather<LBMD_STORE_F16><<<blocks, 256, 0, s>>>(mem, beads, nb, live, cur); break;
    case LBMD_STORE_BF16: k_ens_gather<LBMD_STORE_BF16><<<blocks, 256, 0, s>>>(mem, beads, nb, live, cur); break;
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

cudaError_t launch_ens_md_cycle(const EnsMember *mem, const int *chains, int count, int threads,
                                int max_n, const int *live, bool alone, int priority, cudaStream_t s) {
  if (count <= 0) return cudaSuccess;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)count);
  cfg.blockDim = dim3((unsigned)threads);
  cfg.dynamicSmemBytes = md_smem_bytes(max_n);
  if (alone) {
    const cudaError_t e = md_alone_bytes(&cfg.dynamicSmemBytes);
    if (e != cudaSuccess) return e;
  }
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributePriority;
  attr[0].val.priority = priority;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  if (threads <= 512) return cudaLaunchKernelEx(&cfg, k_ens_md_cycle<512>, mem, chains, live);
  if (threads <= 768) return cudaLaunchKernelEx(&cfg, k_ens_md_cycle<768>, mem, chains, live);
  return cudaLaunchKernelEx(&cfg, k_ens_md_cycle<1024>, mem, chains, live);
}

// Ensemble sum part of the spread, after every MD group: one thread per
// (realisation, bead, corner) entry as in k_ens_gather, adding the entry's
// share to its owner's fixed-point sum (spread_add); k_ens_spread_finalize then
// writes every entry's record (spread_record) to rec[entry].
__global__ void __launch_bounds__(256)
    k_ens_spread_accum(const EnsMember *__restrict__ mem, const int2 *__restrict__ beads, int nb,
                       const int *__restrict__ live) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  const int slot = e >> 3, k = e & 7;
  if (slot >= nb) return;
  const int2 mi = beads[slot];
  if (mi.x < 0 || !live[mi.x]) return;
  const ChainArgs &a = mem[mi.x].a;
  if (a.owner == nullptr) return;  // no solvent: nothing to spread
  spread_add(a, 8 * mi.y + k, a.J[mi.y]);
}
__global__ void __launch_bounds__(256)
    k_ens_spread_finalize(const EnsMember *__restrict__ mem, const int2 *__restrict__ beads, int nb,
                          const int *__restrict__ live, float4 *__restrict__ rec) {
  asm volatile("griddepcontrol.wait;" ::: "memory");  // every share
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >> 3 >= nb) return;
  const int2 mi = beads[e >> 3];
  if (mi.x < 0 || !live[mi.x]) return;
  rec[e] = spread_record(mem[mi.x].a, 8 * mi.y + (e & 7));
}

cudaError_t launch_ens_spread_sum(const EnsMember *mem, const int2 *beads, int nb, const int *live,
                                  float4 *rec, cudaStream_t s) {
  if (nb <= 0) return cudaSuccess;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((8 * nb + 255) / 256);
  cfg.blockDim = dim3(256);
  cfg.stream = s;
  const cudaError_t e = cudaLaunchKernelEx(&cfg, k_ens_spread_accum, mem, beads, nb, live);
  if (e != cudaSuccess || !rec) return e;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k_ens_spread_finalize, mem, beads, nb, live, rec);
}

template <int S>
static void ens_spread_as(const EnsMember *mem, const int2 *beads, int nb, const int *live, int *live_next,
                          int cur, const long long *max_steps, const float4 *rec, cudaStream_t s) {
  const int blocks = nb > 0 ? (8 * nb + 255) / 256 : 1;
  if (rec)
    k_ens_spread<S, false><<<blocks, 256, 0, s>>>(mem, beads, nb, live, live_next, cur, max_steps, rec);
  else
    k_ens_spread<S, true><<<blocks, 256, 0, s>>>(mem, beads, nb, live, live_next, cur, max_steps, rec);
}

cudaError_t launch_ens_spread(int storage, const EnsMember *mem, const int2 *beads, int nb,
                              const int *live, int *live_next, int cur,
                              const long long *max_steps, const float4 *rec, cudaStream_t s) {
  switch (storage) {
    case LBMD_STORE_F32: ens_spread_as<LBMD_STORE_F32>(mem, beads, nb, live, live_next, cur, max_steps, rec, s); break;
    case LBMD_STORE_F16: ens_spread_as<LBMD_STORE_F16>(mem, beads, nb, live, live_next, cur, max_steps, rec, s); break;
    case LBMD_STORE_BF16: ens_spread_as<LBMD_STORE_BF16>(mem, beads, nb, live, live_next, cur, max_steps, rec, s); break;
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

__global__ void k_ens_status(const EnsMember *__restrict__ mem, int count, DevStatus *__restrict__ out) {
  const int m = blockIdx.x * blockDim.x + threadIdx.x;
  if (m < count) out[m] = *mem[m].a.status;
}

cudaError_t launch_ens_status(const EnsMember *mem, int count, DevStatus *out, cudaStream_t s) {
  k_ens_status<<<(count + 127) / 128, 128, 0, s>>>(mem, count, out);
  return cudaGetLastError();
}

__global__ void k_read_beads(const float4 *pos, const float4 *pos_lo, const float4 *vel, int N,
                             int ox, int oy, int oz, double *dpos, double *dvel) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= N) return;
  if (dpos) {
    const float4 r = pos[i];
    const float4 l = pos_lo ? pos_lo[i] : make_float4(0, 0, 0, 0);
    dpos[3 * i] = (double)ox + (double)r.x + (double)l.x;
    dpos[3 * i + 1] = (double)oy + (double)r.y + (double)l.y;
    dpos[3 * i + 2] = (double)oz + (double)r.z + (double)l.z;
  }
  if (dvel) {
    const float4 v = vel[i];
    dvel[3 * i] = v.x;
    dvel[3 * i + 1] = v.y;
    dvel[3 * i + 2] = v.z;
  }
}

cudaError_t launch_read_beads(const float4 *pos, const float4 *pos_lo, const float4 *vel, int N,
                              int ox, int oy, int oz, double *dpos, double *dvel, cudaStream_t s) {
  if (N <= 0) return cudaSuccess;
  k_read_beads<<<(N + 255) / 256, 256, 0, s>>>(pos, pos_lo, vel, N, ox, oy, oz, dpos, dvel);
  return cudaGetLastError();
}

// The block of lbmd_read_beads_async: the status word at offset 0, then the
// unwrapped positions and the velocities (3N doubles each) from offset 32.
__global__ void k_bead_block(const float4 *pos, const float4 *pos_lo, const float4 *vel, int N,
                             int ox, int oy, int oz, const DevStatus *st, char *out) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i == 0) {
    lbmd_status_word *w = (lbmd_status_word *)out;
    w->step = st->step;
    w->t_transloc = st->t_transloc;
    w->n_trans = st->n_trans;
    // a box without beads has no apply kernel to fold the population flag in
    w->state = st->state == LBMD_RUNNING && st->pop_bad ? LBMD_NAN : st->state;
    // the header's padding reads zero: every byte of the block is defined
    for (size_t b = sizeof(lbmd_status_word); b < kBeadBlockHeader; b += sizeof(int)) *(int *)(out + b) = 0;
  }
  if (i >= N) return;
  double *dpos = (double *)(out + kBeadBlockHeader), *dvel = dpos + 3 * (size_t)N;
  const float4 r = pos[i], l = pos_lo[i], v = vel[i];
  dpos[3 * i] = (double)ox + (double)r.x + (double)l.x;
  dpos[3 * i + 1] = (double)oy + (double)r.y + (double)l.y;
  dpos[3 * i + 2] = (double)oz + (double)r.z + (double)l.z;
  dvel[3 * i] = v.x;
  dvel[3 * i + 1] = v.y;
  dvel[3 * i + 2] = v.z;
}

const void *bead_block_kernel() { return reinterpret_cast<const void *>(&k_bead_block); }

cudaError_t launch_bead_block(const ChainArgs &a, const DevStatus *st, void *out, cudaStream_t s) {
  const int n = a.N > 0 ? a.N : 1;
  k_bead_block<<<(n + 255) / 256, 256, 0, s>>>(a.pos, a.pos_lo, a.vel, a.N, a.ox, a.oy, a.oz, st,
                                               (char *)out);
  return cudaGetLastError();
}

cudaError_t launch_read_bead_aux(const float4 *ui, const float4 *J, int N, double *dui,
                                 double *dJ, cudaStream_t s) {
  if (N <= 0) return cudaSuccess;
  k_read_beads<<<(N + 255) / 256, 256, 0, s>>>(ui, nullptr, J, N, 0, 0, 0, dui, dJ);
  return cudaGetLastError();
}

}  // namespace lbmd
