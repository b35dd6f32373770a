"""Walls where the stream-collides' test for "beside a wall" can go wrong: the
wall at the box's edge, wrapping around it, several layers thick, a pore at a
corner, together with y-walls, widths whose rows straddle the 64-node blocks of
16-bit storage, and a box beyond the L2 cache (solid nodes written).  Every
population against the FP64 oracle after three steps from a random flow.

Tolerances as the population tests of the same storage: 1e-5 relative per FP32
step; 16-bit deviations round to half an ulp of |h| <= 0.05 three times over,
relative to the smallest weight 1/36 (2^-12 0.05 36 3 = 1.4e-3 for FP16)."""
import numpy as np
import pytest

import oracle
import seeded_inputs as si

pytestmark = pytest.mark.gpu

CASES = [
    dict(nx=6, ny=5, nz=4, wall_x=5, wall_thickness=2, pore_d=1, pore_y0=0, pore_z0=0),
    dict(nx=8, ny=6, nz=5, wall_x=0, wall_thickness=1, pore_d=2, pore_y0=4, pore_z0=3, y_walls=1),
    dict(nx=2, ny=3, nz=3, wall_x=1, wall_thickness=1, pore_d=1),
    dict(nx=3, ny=4, nz=2, wall_x=2, wall_thickness=2, pore_d=0),
    dict(nx=40, ny=6, nz=3, wall_x=38, wall_thickness=9, pore_d=3),
    dict(nx=96, ny=7, nz=5, wall_x=63, wall_thickness=1, pore_d=3, y_walls=1),
    dict(nx=130, ny=3, nz=3, wall_x=64, wall_thickness=3, pore_d=1),
    dict(nx=33, ny=9, nz=4, wall_x=32, wall_thickness=1, pore_d=3),
]


@pytest.mark.parametrize("streaming", ["pull", "aa"])
@pytest.mark.parametrize("storage,tol", [("f32", 3e-5), ("f16", 1.4e-3)])
@pytest.mark.parametrize("case", range(len(CASES)))
def test_walls_against_the_oracle(case, storage, tol, streaming):
    _compare(dict(CASES[case], tau=0.8, body_force=(1e-5, 0, 0)), storage, tol, streaming)


@pytest.mark.parametrize("storage,tol", [("f32", 3e-5), ("f16", 1.4e-3)])
def test_thin_wall_in_a_box_beyond_l2(storage, tol):
    n = 1 if storage == "f32" else 2
    _compare(dict(nx=160, ny=80, nz=72 * n, wall_x=80, wall_thickness=2, pore_d=5), storage, tol, "pull")


def _compare(p, storage, tol, streaming):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_0710_1272_gb300 as lb
    rho, u = si.random_flow((p["nz"], p["ny"], p["nx"]), seed=11, rho_spread=0.02, u_max=0.02)
    sim = lb.Simulation(dict(p, storage=storage, streaming=streaming), init_rho=rho, init_u=u)
    orc = oracle.OracleSim(p, init_rho=rho, init_u=u)
    sim.step(3)
    orc.step(3)
    f, o = sim.populations(), orc.populations()
    m = o != 0
    assert np.all(f[~m] == 0)
    assert np.max(np.abs(f[m] - o[m]) / np.abs(o[m])) < tol


@pytest.mark.parametrize("nx,offset", [(32, 0), (32, 1), (33, 0), (33, 1)])
def test_population_readout_alignment(nx, offset):
    """Paired 8-byte stores only where the row length and the caller's memory
    allow them: the same values wherever the caller wants them."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_0710_1272_gb300 as lb
    p = dict(nx=nx, ny=5, nz=3, wall_x=16, pore_d=3, storage="f16", init_tg_amp=0.02)
    sim = lb.Simulation(p)
    sim.step(2)
    n = 19 * nx * 5 * 3
    buf = torch.full((n + 3,), 7.0, dtype=torch.float32, device="cuda")
    lb.lbmd_read_populations(sim.ctx, buf[offset:].data_ptr(), 1)
    torch.cuda.synchronize()
    got = buf.cpu().numpy()
    assert np.array_equal(got[offset:offset + n].reshape(19, 3, 5, nx), sim.populations())
    assert np.all(got[:offset] == 7.0) and np.all(got[offset + n:] == 7.0)
