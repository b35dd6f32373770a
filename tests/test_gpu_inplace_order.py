"""In-place against two-buffer streaming with a chain, bit for bit, on either side of the size from which a
two-buffer stream-collide starts beside the bead gather: an in-place one has to wait for it."""
import numpy as np
import pytest

import paper_0710_1272_gb300 as lb

pytestmark = pytest.mark.gpu


def _chain(n, nx, ny, nz):
    """Zigzag along x whose beads lie about the planes z = 0 and z = nz - 1, which the first and the last
    blocks of the stream-collide update."""
    pos = np.zeros((n, 3))
    pos[:, 0] = 4.0 + 1.1 * np.arange(n)
    pos[:, 1] = 0.5 * ny
    pos[:, 2] = np.where(np.arange(n) % 2, 0.25, -0.2295)  # bonds of 1.2
    return pos


@pytest.mark.parametrize("storage,shape", [
    ("f32", (128, 112, 109)), ("f32", (128, 112, 112)), ("f32", (128, 112, 128)), ("f32", (128, 112, 129)),
    ("f16", (160, 144, 135)), ("f16", (160, 144, 160)), ("f16", (161, 144, 159)), ("bf16", (160, 144, 160))])
def test_in_place_equals_pull_with_a_chain(storage, shape):
    nx, ny, nz = shape
    n = 100
    p = dict(nx=nx, ny=ny, nz=nz, n_beads=n, lj_sigma=1.0, lj_eps=2e-3, storage=storage, init_tg_amp=0.02, seed=11)
    a = lb.Simulation(dict(p, streaming="aa"), init_pos=_chain(n, nx, ny, nz))
    b = lb.Simulation(p, init_pos=_chain(n, nx, ny, nz))
    for steps in (1, 1, 16, 3, 2):
        a.step(steps)
        b.step(steps)
        for x, y in zip(a.beads() + a.bead_aux(), b.beads() + b.bead_aux()):
            np.testing.assert_array_equal(x, y)
    np.testing.assert_array_equal(a.populations(), b.populations())
    assert a.status()["state"] == lb.RUNNING
