"""Ensembles on either side of the sizes at which short chains get an SM to themselves, against single boxes."""
import numpy as np
import pytest

import paper_0710_1272_gb300 as lb

pytestmark = pytest.mark.gpu


def _line(n, ny, nz):
    pos = np.zeros((n, 3))
    pos[:, 0] = 2.0 + 1.1 * np.arange(n)
    pos[:, 1] = 0.5 * ny
    pos[:, 2] = 0.5 * nz + np.where(np.arange(n) % 2, 0.25, -0.2295)  # bonds of 1.2
    return pos


# populations of a step: 55, 63, 394 and 404 MB; the last member's chain takes a block of more than 128 threads
@pytest.mark.parametrize("storage,shape", [
    ("f32", (64, 44, 43)), ("f16", (128, 67, 32)), ("f16", (160, 90, 120)), ("f32", (160, 60, 92))])
def test_short_chains_alone_equal_single_boxes(storage, shape):
    nx, ny, nz = shape
    lengths = [2, 33, 96] if nx < 100 else [20, 64, 130]
    members = [dict(nx=nx, ny=ny, nz=nz, n_beads=n, lj_sigma=1.0, lj_eps=2e-3, seed=n, storage=storage, kappa_phi=0.01)
               for n in lengths]
    starts = [_line(n, ny, nz) for n in lengths]
    ens = lb.Ensemble(members, starts)
    ens.step(19)
    steps = ens.results()["steps"]  # a chain that meets itself across the box ends its realisation
    for k, (m, start) in enumerate(zip(members, starts)):
        one = lb.Simulation(m, init_pos=start)
        one.step(int(steps[k]))
        for x, y in zip(ens.beads(k), one.beads()):
            np.testing.assert_array_equal(x, y)
        np.testing.assert_array_equal(ens.populations(k), one.populations())


# 594 and 627 MB: the gather beside the stream-collide and the forces through records from 600 MB on
@pytest.mark.parametrize("storage,shape", [("f32", (96, 102, 133)), ("f32", (96, 102, 141)), ("f16", (161, 128, 134))])
def test_large_ensembles_equal_single_boxes(storage, shape):
    nx, ny, nz = shape
    members = [dict(nx=nx, ny=ny, nz=nz, n_beads=n, lj_sigma=1.0, lj_eps=2e-3, seed=n, storage=storage) for n in (5, 40, 75)]
    starts = [_line(m["n_beads"], ny, nz) for m in members]
    ens = lb.Ensemble(members, starts)
    ens.step(18)
    steps = ens.results()["steps"]
    for k, (m, start) in enumerate(zip(members, starts)):
        one = lb.Simulation(m, init_pos=start)
        one.step(int(steps[k]))
        for x, y in zip(ens.beads(k), one.beads()):
            np.testing.assert_array_equal(x, y)
        np.testing.assert_array_equal(ens.populations(k), one.populations())
