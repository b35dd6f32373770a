// lb_noalloc.cu -- one D3Q19 stream-collide step on caller-owned populations
// that allocates nothing: no context, no workspace, no cudaMalloc.
//
// Who needs it: code that cannot allocate device memory -- a caller whose
// device memory is entirely handed out by another framework's pool, code that
// runs while another thread captures a CUDA graph in global capture mode
// (where cudaMalloc is prohibited), or a real-time loop that must not touch
// the allocator -- but does own two population buffers and wants the solvent
// update of the coupled step (no beads).
//
// One kernel and no memory besides the caller's input and output: whether a
// node or its neighbour is solid is computed from the Sec. III geometry, for
// the few nodes beside a wall.  (Two more kernels used to build a bitfield and
// tile flags in a fixed device array on every call, 9 us and two launches of a
// 73 us call on 160x96x96, and calls on different streams raced on it.)
// The box stays limited to the size that array had room for.
#include <cuda_runtime.h>

#include "lbmd_common.cuh"

namespace lbmd {
namespace {

constexpr int kNoAllocMaxTiles = 1 << 20;  // ny nz ceil(nx / 32): 2^25 nodes, 32-bit offsets

struct GeoParams {
  int nx, ny, nz;
  WallGeom wall;
};

// Which of the node itself (bit 0) and its neighbours x + c_p (bit p) are solid.
__device__ __forceinline__ uint32_t solid_around(const GeoParams &q, int x, int y, int z) {
  const WallGeom &w = q.wall;
  int dx = x - w.wall_x;  // layers after the first one, around the box
  if (dx < 0) dx += q.nx;
  const bool layer = w.wall_x >= 0 && (dx <= w.wall_t || dx == q.nx - 1);
  const bool rows = w.y_walls && (y <= 1 || y >= q.ny - 2);
  if (!layer && !rows) return 0u;
  // solid along each axis at offsets -1, 0, +1
  bool in[3], row[3], py[3], pz[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    int a = dx + k - 1;
    a = a < 0 ? a + q.nx : (a >= q.nx ? a - q.nx : a);
    in[k] = w.wall_x >= 0 && a < w.wall_t;
    const int b = k == 0 ? wrap_m1(y, q.ny) : (k == 2 ? wrap_p1(y, q.ny) : y);
    const int c = k == 0 ? wrap_m1(z, q.nz) : (k == 2 ? wrap_p1(z, q.nz) : z);
    row[k] = w.y_walls && (b == 0 || b == q.ny - 1);
    py[k] = b >= w.pore_y0 && b < w.pore_y0 + w.pore_d;
    pz[k] = c >= w.pore_z0 && c < w.pore_z0 + w.pore_d;
  }
  uint32_t s = 0u;
#pragma unroll
  for (int p = 0; p < kQ; ++p)
    if (row[1 + cy(p)] || (in[1 + cx(p)] && !(py[1 + cy(p)] && pz[1 + cz(p)]))) s |= 1u << p;
  return s;
}

// Collide-then-push form of Eq. 5 on absolute populations:
//   f*_p(x) = f_p - (f_p - f_eq,p(rho, u)) / tau + S_p(g),
//   f_p(x + c_p, t+1) = f*_p(x) if x + c_p is fluid, else f_opp(p)(x, t+1) = f*_p(x).
// Solid nodes of the output are set to zero.  Bound by HBM (19 loads, 19
// stores per node, those for c_x = +-1 shifted by a node); 32-bit offsets and
// one reciprocal per node, where 64-bit offsets, three divisions and per-tile
// flags had made it a kernel of 60 us at 160x96x96 (33 us of traffic): the whole
// call took 71.9 us, now 42.5.
template <int FORCING>
__global__ void __launch_bounds__(256, 5) k_noalloc_step(GeoParams q, float omega, float gx, float gy,
                                                         float gz, const float *__restrict__ fin,
                                                         float *__restrict__ fout) {
  const int x = blockIdx.x * 32 + threadIdx.x;
  const int y = blockIdx.y * 8 + threadIdx.y;
  const int z = blockIdx.z;
  if (x >= q.nx || y >= q.ny) return;
  const int nx = q.nx, ny = q.ny, nz = q.nz;
  const int V = nx * ny * nz;
  const int self = (z * ny + y) * nx + x;
  float f[kQ];
#pragma unroll
  for (int p = 0; p < kQ; ++p) f[p] = __ldg(fin + (p * V + self));
  const uint32_t solid = solid_around(q, x, y, z);
  if (solid & 1u) {
#pragma unroll
    for (int p = 0; p < kQ; ++p) fout[p * V + self] = 0.f;
    return;
  }
  float rho = f[0], jx = 0.f, jy = 0.f, jz = 0.f;
#pragma unroll
  for (int p = 1; p < kQ; ++p) {
    rho += f[p];
    if (cx(p)) jx += cx(p) > 0 ? f[p] : -f[p];
    if (cy(p)) jy += cy(p) > 0 ? f[p] : -f[p];
    if (cz(p)) jz += cz(p) > 0 ? f[p] : -f[p];
  }
  if (FORCING == LBMD_FORCING_GUO) {
    jx += 0.5f * gx;
    jy += 0.5f * gy;
    jz += 0.5f * gz;
  }
  const float inv = 1.0f / rho;
  const float ux = jx * inv, uy = jy * inv, uz = jz * inv;
  const float base = 1.0f - 1.5f * (ux * ux + uy * uy + uz * uz);
  const float gu = gx * ux + gy * uy + gz * uz;
  const float kguo = 1.0f - 0.5f * omega;
  // source of direction p, c_p . u = cu
  const auto source = [&](int p, float cu) {
    const float cg = cx(p) * gx + cy(p) * gy + cz(p) * gz;
    return FORCING == LBMD_FORCING_GUO ? kguo * wq(p) * (3.0f * (cg - gu) + 9.0f * cu * cg)
                                       : 3.0f * wq(p) * cg;
  };
  // opposite directions p, p + 1 (odd p) share the even part of the equilibrium
  f[0] = f[0] - omega * (f[0] - wq(0) * rho * base) + source(0, 0.f);
#pragma unroll
  for (int p = 1; p < kQ; p += 2) {
    const float cu = cx(p) * ux + cy(p) * uy + cz(p) * uz, wr = wq(p) * rho;
    const float even = wr * (base + 4.5f * cu * cu), odd = 3.0f * wr * cu;
    f[p] = f[p] - omega * (f[p] - (even + odd)) + source(p, cu);
    f[p + 1] = f[p + 1] - omega * (f[p + 1] - (even - odd)) + source(p + 1, -cu);
  }
  const int xm = wrap_m1(x, nx), xp = wrap_p1(x, nx), ym = wrap_m1(y, ny), yp = wrap_p1(y, ny);
  const int zm = wrap_m1(z, nz), zp = wrap_p1(z, nz);
#pragma unroll
  for (int p = 0; p < kQ; ++p) {
    const int xd = cx(p) == 1 ? xp : (cx(p) == -1 ? xm : x);
    const int yd = cy(p) == 1 ? yp : (cy(p) == -1 ? ym : y);
    const int zd = cz(p) == 1 ? zp : (cz(p) == -1 ? zm : z);
    const int to = p * V + ((zd * ny + yd) * nx + xd), back = opp(p) * V + self;
    fout[((solid >> p) & 1u) ? back : to] = f[p];
  }
}

}  // namespace
}  // namespace lbmd

using namespace lbmd;

extern "C" int lbmd_lb_step_noalloc(const lbmd_params *p, const float *f_in, float *f_out,
                                    void *cuda_stream) {
  if (!p || !f_in || !f_out) return LBMD_EINVAL;
  if (f_in == f_out) return LBMD_EINVAL;
  if (p->nx < 1 || p->ny < 1 || p->nz < 1 || p->nz > 65535) return LBMD_EINVAL;
  if (!(p->tau > 0.5) || !(p->rho0 > 0)) return LBMD_EINVAL;
  // FP32 solvent only: no bead state to keep, no step counter for the noise
  if (p->storage != LBMD_STORE_F32 || p->n_beads != 0 || p->kT_fluid != 0.0) return LBMD_EUNSUPPORTED;
  if (p->forcing != LBMD_FORCING_PAPER && p->forcing != LBMD_FORCING_GUO) return LBMD_EINVAL;
  if (p->wall_x < -1 || p->wall_x >= p->nx) return LBMD_EINVAL;
  if (p->y_walls != 0 && p->y_walls != 1) return LBMD_EINVAL;
  GeoParams q;
  q.nx = p->nx;
  q.ny = p->ny;
  q.nz = p->nz;
  q.wall = WallGeom{p->wall_x, p->wall_thickness, 0, 0, 0, p->y_walls};
  if (p->wall_x >= 0) {
    if (p->wall_thickness < 1 || p->wall_thickness >= p->nx) return LBMD_EINVAL;
    if (p->pore_d < 0 || p->pore_d > p->ny || p->pore_d > p->nz) return LBMD_EINVAL;
    q.wall.pore_d = p->pore_d;
    q.wall.pore_y0 = p->pore_y0 >= 0 ? p->pore_y0 : (p->ny - p->pore_d) / 2;
    q.wall.pore_z0 = p->pore_z0 >= 0 ? p->pore_z0 : (p->nz - p->pore_d) / 2;
    if (q.wall.pore_y0 + p->pore_d > p->ny || q.wall.pore_z0 + p->pore_d > p->nz) return LBMD_EINVAL;
  }
  const int ntx = (q.nx + 31) / 32;
  const long long tiles = (long long)q.ny * q.nz * ntx;
  if (tiles > kNoAllocMaxTiles) return LBMD_ESIZE;  // box beyond the limit
  if ((q.ny + 7) / 8 > 65535) return LBMD_EINVAL;   // grid y of the step kernel (ny <= 524280)

  // launched with cudaLaunchKernelEx, whose return value is the status of
  // that launch alone (not an error left behind by unrelated earlier work)
  cudaLaunchConfig_t cfg = {};
  cfg.stream = (cudaStream_t)cuda_stream;
  cfg.blockDim = dim3(32, 8);
  cfg.gridDim = dim3(ntx, (q.ny + 7) / 8, q.nz);
  const float omega = (float)(1.0 / p->tau);
  const float gx = (float)p->body_force[0], gy = (float)p->body_force[1], gz = (float)p->body_force[2];
  const cudaError_t e =
      p->forcing == LBMD_FORCING_GUO
          ? cudaLaunchKernelEx(&cfg, k_noalloc_step<LBMD_FORCING_GUO>, q, omega, gx, gy, gz, f_in, f_out)
          : cudaLaunchKernelEx(&cfg, k_noalloc_step<LBMD_FORCING_PAPER>, q, omega, gx, gy, gz, f_in, f_out);
  return e == cudaSuccess ? LBMD_OK : LBMD_ECUDA;
}
