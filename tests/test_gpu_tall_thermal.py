"""A fluctuating FP32 solvent with more rows than one launch of its two-node kernel covers."""
import numpy as np
import pytest

import paper_0710_1272_gb300 as lb

pytestmark = pytest.mark.gpu


# just below and above the 65535 x 4 rows of one launch, and the largest ny that the other kernels take
@pytest.mark.parametrize("ny", [262140, 262141, 524280])
def test_tall_box_equals_in_place(ny):
    p = dict(nx=3, ny=ny, nz=2, n_beads=0, kT_fluid=1e-4, tau=0.8, seed=5, init_tg_amp=0.01)
    a, b = lb.Simulation(p), lb.Simulation(dict(p, streaming="aa"))
    a.step(3)
    b.step(3)
    np.testing.assert_array_equal(a.populations(), b.populations())
