"""The normals of the FP32 thermal source (box_muller_t) over all 2^23 values of either uniform, one and two
nodes at a time, against FP64 and against the CUDA library's functions."""
import ctypes
import os
import subprocess

import pytest

from paper_0710_1272_gb300 import build as lb_build

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include <cstdio>
#include "lb_collide.cuh"
using namespace lbmd;

// sums over all k < 2^23 (u1 from k, u2 from a permutation of k): 0, 1 relative errors squared (ours, library's);
// 2, 3 largest errors over the radius; 4 how often one and two nodes at a time differ
__global__ void k_compare(unsigned salt, double *out) {
  double e2 = 0, l2 = 0;
  float em = 0, lm = 0;
  unsigned differ = 0;
  for (unsigned k = blockIdx.x * blockDim.x + threadIdx.x; k < 1u << 23; k += gridDim.x * blockDim.x) {
    const unsigned q = (k * 2654435761u + salt) & ((1u << 23) - 1);
    const unsigned x1[2] = {k << 9, ((k + 1) << 9)}, x2[2] = {q << 9, ((q + 12345u) << 9)};
    float a1, a2;
    box_muller_t<Ops1>(uniform23_t<Ops1>(x1), uniform23_t<Ops1>(x2), a1, a2);
    float2 b1, b2;
    box_muller_t<Ops2>(uniform23_t<Ops2>(x1), uniform23_t<Ops2>(x2), b1, b2);
    float c1, c2;
    box_muller_t<Ops1>(uniform23_t<Ops1>(x1 + 1), uniform23_t<Ops1>(x2 + 1), c1, c2);
    differ += __float_as_int(a1) != __float_as_int(b1.x) || __float_as_int(a2) != __float_as_int(b2.x) ||
              __float_as_int(c1) != __float_as_int(b1.y) || __float_as_int(c2) != __float_as_int(b2.y);
    const float u1 = uniform23(x1[0]), u2 = uniform23(x2[0]);
    const float rad = sqrtf(-2.0f * logf(u1));
    float sn, cs;
    sincospif(2.0f * u2, &sn, &cs);
    const double r = sqrt(-2.0 * log((double)u1));
    double ds, dc;
    sincospi(2.0 * (double)u2, &ds, &dc);
    const double w[2] = {r * dc, r * ds};
    const float ours[2] = {a1, a2}, lib[2] = {rad * cs, rad * sn};
    for (int n = 0; n < 2; ++n) {
      const double eo = (ours[n] - w[n]) / w[n], el = (lib[n] - w[n]) / w[n];
      e2 += eo * eo;
      l2 += el * el;
      em = fmaxf(em, (float)(fabs(ours[n] - w[n]) / r));
      lm = fmaxf(lm, (float)(fabs(lib[n] - w[n]) / r));
    }
  }
  atomicAdd(out, e2);
  atomicAdd(out + 1, l2);
  atomicMax((unsigned long long *)(out + 2), (unsigned long long)__double_as_longlong((double)em));
  atomicMax((unsigned long long *)(out + 3), (unsigned long long)__double_as_longlong((double)lm));
  atomicAdd(out + 4, (double)differ);
}
extern "C" int compare(unsigned salt, double *host) {
  double *d;
  if (cudaMalloc(&d, 5 * sizeof(double)) != cudaSuccess) return 1;
  cudaMemset(d, 0, 5 * sizeof(double));
  k_compare<<<304, 256>>>(salt, d);
  const int e = cudaMemcpy(host, d, 5 * sizeof(double), cudaMemcpyDeviceToHost) != cudaSuccess;
  cudaFree(d);
  return e;
}
"""


@pytest.fixture(scope="module")
def compare(tmp_path_factory):
    d = tmp_path_factory.mktemp("box_muller")
    src, lib = d / "compare.cu", d / "libcompare.so"
    src.write_text(SOURCE)
    subprocess.run([lb_build.nvcc(), *lb_build.FLAGS, *lb_build.ARCH, "-I", lb_build.CSRC, "-I",
                    os.path.join(lb_build.ROOT, "include"), "-shared", str(src), "-o", str(lib)], check=True)
    return ctypes.CDLL(str(lib))


# Bounds: a normal is a rounded radius times a rounded cosine, rounded once more; three errors of up to half a
# unit in the last place, 2^-24 relative each, are 1.8e-7 at most and, spread evenly, 3^(1/2) 2^-24 / 3^(1/2) =
# 6e-8 in the root mean square.  The library's functions set the rest: not less exact than they.
@pytest.mark.parametrize("salt", [0, 777, 4194304, 8388607])
def test_normals(compare, salt):
    out = (ctypes.c_double * 5)()
    assert compare.compare(ctypes.c_uint(salt), out) == 0
    ours, lib, worst, worst_lib, differ = out
    rms, rms_lib = ((s / 2**24) ** 0.5 for s in (ours, lib))
    print(f"rms {rms:.4e} library {rms_lib:.4e}, largest of the radius {worst:.3e} library {worst_lib:.3e}")
    assert differ == 0
    assert rms <= 6e-8 and worst <= 1.8e-7
    assert rms <= rms_lib
