"""The MD block at the sizes where its constraint solve and its force lists
change form: chain lengths around whole warps, around the row counts of the
one-warp tridiagonal solve (160, 416, 544 rows; halved systems from 513 beads
on) and around the block's register classes, each against the FP64 oracle.

Tolerances as the parity tests of the same quantities: beads within 2e-5 after
two steps (1024-bead chain), 1e-5 after three (list fallbacks)."""
import numpy as np
import pytest

import oracle
import seeded_inputs as si

pytestmark = pytest.mark.gpu


def _pair(p, pos, bonds=None):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_0710_1272_gb300 as lb
    sim = lb.Simulation(p, init_pos=pos, bonds=bonds)
    orc = oracle.OracleSim(p, init_pos=pos, bonds=bonds)
    return sim, orc


@pytest.mark.parametrize("n", [2, 3, 32, 33, 65, 97, 161, 162, 417, 418, 480, 481, 512, 513, 736, 768, 833,
                               834, 993])
def test_chain_lengths_around_the_solve_sizes(n):
    p = dict(si.paper_translocation(1, n_beads=n), nx=128, ny=64, nz=64, wall_x=32, lj_eps=2e-3,
             hydrodynamics=0, kappa_phi=0.05 if n % 2 else 0.0)
    pos = si.saw_chain(p, 1)
    sim, orc = _pair(p, pos)
    sim.step(2)
    orc.step(2)
    r, v = sim.beads()
    assert np.abs(r - orc.beads()[0]).max() < 2e-5
    assert np.abs(v - orc.beads()[1]).max() < 2e-5
    assert sim.status()["state"] == 0 and sim.solver_stats()["failed_steps"] == 0
    b = np.linalg.norm(np.diff(r, axis=0), axis=1)
    assert np.abs(b - 1.2).max() < 2e-6  # a few roundings of a unit coordinate in FP32


def test_chain_with_a_solvent_one_past_a_warp():
    """65 beads: the last bond lies in a warp of its own."""
    p = dict(si.small_translocation(3, n_beads=65), nx=64, ny=32, nz=32, wall_x=32, lj_eps=2e-3)
    pos = si.saw_chain(p, 3)
    sim, orc = _pair(p, pos)
    sim.step(3)
    orc.step(3)
    assert np.abs(sim.beads()[0] - orc.beads()[0]).max() < 2e-5
    assert np.abs(sim.populations() - orc.populations()).max() < 2e-5 / 3


def test_dense_beads_take_the_lists_of_their_own():
    """64 free beads on a grid (sigma = 0.65: every bead has up to 32 partners
    within r_c + skin): more entries than the block's force list holds, none of
    the beads' own lists overflowing."""
    p = dict(si.small_translocation(0, n_beads=64), wall_x=-1, lj_sigma=0.65, lj_eps=1e-3, kT=1e-4)
    k = np.arange(64)
    pos = np.array([10.0, 6.0, 6.0]) + 0.7 * np.stack([k % 4, k // 4 % 4, k // 16], 1)
    nb = (np.zeros(0, np.int32), np.zeros(0, np.int32), np.zeros(0))
    sim, orc = _pair(p, pos, nb)
    sim.step(3)
    orc.step(3)
    assert np.abs(sim.beads()[0] - orc.beads()[0]).max() < 1e-5


def test_beads_with_more_than_31_solid_nodes():
    """Three beads in a 3 x 3 pore through a wall of five layers, off its axis:
    more solid nodes each than the acting-entry mask has bits."""
    p = dict(si.small_translocation(0, n_beads=3), wall_thickness=5, wall_x=12, lj_eps=2e-3)
    pos = np.array([[13.0, 7.4, 7.3], [14.2, 7.4, 7.3], [15.4, 7.4, 7.3]])
    sim, orc = _pair(p, pos)
    sim.step(3)
    orc.step(3)
    assert np.abs(sim.beads()[0] - orc.beads()[0]).max() < 1e-5
