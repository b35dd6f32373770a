"""16-bit populations of boxes about the width from which two nodes share a thread: in place against two
buffers, bit for bit, with the read-outs of populations and fields."""
import numpy as np
import pytest

import paper_0710_1272_gb300 as lb

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("storage", ["f16", "bf16"])
@pytest.mark.parametrize("wall", [False, True])
@pytest.mark.parametrize("nx", [2, 31, 32, 33, 34])
def test_in_place_equals_pull(nx, wall, storage):
    p = dict(nx=nx, ny=90, nz=140000 // (90 * nx) + 1, n_beads=0, storage=storage, tau=0.8, init_tg_amp=0.02,
             body_force=(1e-5, 0.0, 0.0), wall_x=nx // 2 if wall else -1, pore_d=3)
    a, b = lb.Simulation(p), lb.Simulation(dict(p, streaming="aa"))
    for n in (1, 1, 6):
        a.step(n)
        b.step(n)
        f = a.populations()
        assert np.isfinite(f).all()
        np.testing.assert_array_equal(f, b.populations())
        np.testing.assert_array_equal(f, a.populations_device().cpu().numpy().reshape(f.shape))
        for x, y in zip(a.fields(), b.fields()):
            np.testing.assert_array_equal(x, y)
