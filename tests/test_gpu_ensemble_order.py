"""Batches large enough for the stream-collide to set the step: the gather runs
beside it and the owners' forces go through records.  Same bits as single boxes,
each of which is below that size and takes the other order."""
import numpy as np
import pytest

import seeded_inputs as si

pytestmark = pytest.mark.gpu


def _lb():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_0710_1272_gb300 as lb
    return lb


# 19 populations in and out of all nodes: just under and over 240 MB
@pytest.mark.parametrize("storage,copies", [("f32", 9), ("f32", 8), ("f16", 17), ("bf16", 16)])
def test_large_batch_matches_single_boxes(storage, copies):
    lb = _lb()
    specs = [dict(nx=50, ny=61, nz=64, wall_x=25, pore_d=5, n_beads=n, seed=20 + n, lj_eps=2e-3,
                  storage=storage) for n in (3, 70)]
    members = [dict(si.BASE, **specs[k % 2]) for k in range(copies)]
    starts = [si.saw_chain(p, p["seed"]) for p in members]
    nodes = copies * 50 * 61 * 64
    assert (2 * 19 * nodes * (4 if storage == "f32" else 2) >= 240_000_000) == (copies in (9, 17))
    ens = lb.Ensemble(members, starts)
    ens.run(9, check_every=4)   # stops on the cap at an odd step
    ens.run(20, check_every=8)
    for k in (0, 1, copies - 1):
        sim = lb.Simulation(members[k], init_pos=starts[k])
        for _ in range(20):
            if sim.status()["state"] != lb.RUNNING:
                break
            sim.step(1)
        assert np.array_equal(ens.populations(k), sim.populations()), k
        for a, b in zip(ens.beads(k), sim.beads()):
            assert np.array_equal(a, b), k
