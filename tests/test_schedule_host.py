"""Order of a coupled step's kernels, as the host decides it (no GPU)."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CUDA = os.environ.get("CUDA_HOME", "/usr/local/cuda")

PROGRAM = r"""
#include <cstdio>
#include "lbmd_internal.h"
int main() {
  for (int storage = 0; storage < 3; ++storage)
    for (long long nodes = 1000; nodes < 100000000; nodes *= 2)
      std::printf("%d %lld %d %d\n", storage, nodes, lbmd::gather_goes_first(storage, nodes, true),
                  lbmd::gather_goes_first(storage, nodes, false));
}
"""


def test_gather_precedes_an_in_place_stream_collide(tmp_path):
    """In-place streaming overwrites the populations that the bead gather reads: whatever the size of
    the box, its stream-collide has to wait for the gather.  With two buffers only small boxes do."""
    if shutil.which("g++") is None or not os.path.isdir(os.path.join(CUDA, "include")):
        pytest.skip("needs g++ and the CUDA headers")
    src, exe = tmp_path / "order.cpp", tmp_path / "order"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-I", os.path.join(CUDA, "include"), "-I", os.path.join(ROOT, "include"),
                    "-I", os.path.join(ROOT, "paper_0710_1272_gb300", "csrc"), str(src), "-o", str(exe)], check=True)
    rows = [list(map(int, r.split())) for r in subprocess.run([str(exe)], check=True, capture_output=True,
                                                              text=True).stdout.splitlines()]
    assert rows and all(in_place == 1 for _, _, in_place, _ in rows)
    for storage, nodes, _, two in rows:
        assert two == (2 * 19 * nodes * (4 if storage == 0 else 2) < 280_000_000)


def test_the_step_asks_for_that_order():
    text = open(os.path.join(ROOT, "paper_0710_1272_gb300", "csrc", "lbmd_abi.cu")).read()
    step = text[text.index("cudaError_t enqueue_step("):text.index("cudaError_t capture(")]
    wait = step.index("if (gather_goes_first(c->p.storage, c->geo.V, c->aa))")
    assert step.index("launch_gather(") < wait < step.index("cudaStreamWaitEvent(c->own, c->ev_gather, 0)")
    assert step.index("cudaStreamWaitEvent(c->own, c->ev_gather, 0)") < step.index("launch_lb_aa(")
