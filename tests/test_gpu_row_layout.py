"""16-bit populations of odd width: an ensemble, whose rows are not padded, against single boxes, whose rows
are, and against the host read-out of both."""
import numpy as np
import pytest

import paper_0710_1272_gb300 as lb

pytestmark = pytest.mark.gpu


def _zigzag(n, y, z):
    pos = np.zeros((n, 3))
    pos[:, 0] = 2.0 + 1.1 * np.arange(n)
    pos[:, 1] = y
    pos[:, 2] = z + np.where(np.arange(n) % 2, 0.25, -0.2295)  # bonds of 1.2
    return pos


@pytest.mark.parametrize("walls", ["behind", "none", "y"])
@pytest.mark.parametrize("storage", ["f16", "bf16"])
@pytest.mark.parametrize("tuning", [(8, 48, 2, 1), (4, 32, 1, 2), (16, 32, 2, 1)])
def test_odd_ensemble_equals_single_boxes(walls, storage, tuning):
    members, starts = [], []
    for k, (nx, ny, nz) in enumerate(((33, 21, 18), (49, 33, 23), (65, 19, 17))):
        members.append(dict(nx=nx, ny=ny, nz=nz, wall_x=nx - 3 if k and walls == "behind" else -1, pore_d=3,
                            y_walls=int(walls == "y"), n_beads=10 + 5 * k, lj_sigma=1.0,
                            lj_eps=2e-3, seed=k + 1, storage=storage, tau=0.8))
        starts.append(_zigzag(10 + 5 * k, ny // 2, nz // 2))
    ens = lb.Ensemble(members, starts)
    ens.set_tuning(*tuning)
    ens.step(20)
    steps = ens.results()["steps"]  # a chain on the far side of its wall ends its realisation
    for k, (m, start) in enumerate(zip(members, starts)):
        one = lb.Simulation(m, init_pos=start)
        one.step(int(steps[k]))
        np.testing.assert_array_equal(ens.populations(k), one.populations())
        for x, y in zip(ens.beads(k), one.beads()):
            np.testing.assert_array_equal(x, y)
