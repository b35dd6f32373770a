"""In-place streaming in 16-bit storage by pairs of nodes (boxes of 2^17 nodes or
more): the same bits as pull streaming after every step, widths even and odd, walls
at either half of a word, the box's edges and the pore included."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

BOXES = [
    dict(nx=64, ny=64, nz=32),                                            # 2^17 nodes, the smallest
    dict(nx=67, ny=45, nz=50),                                            # odd rows
    dict(nx=1, ny=363, nz=363),                                           # a row of one node
    dict(nx=96, ny=41, nz=37, y_walls=1),
    dict(nx=256, ny=23, nz=24, wall_x=127, pore_d=5),                     # wall in the second half
    dict(nx=257, ny=23, nz=24, wall_x=256, pore_d=3),                     # wall in a row's lone node
    dict(nx=257, ny=23, nz=24, wall_x=0, wall_thickness=3, pore_d=4, y_walls=1),
    dict(nx=255, ny=23, nz=24, wall_x=100, pore_d=5),                     # odd step by single nodes
]


@pytest.mark.parametrize("storage,force", [("f16", 0.0), ("bf16", 0.0), ("f16", 1e-5)])
@pytest.mark.parametrize("box", range(len(BOXES)))
def test_inplace_pairs_match_pull(box, storage, force):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_0710_1272_gb300 as lb

    p = dict(BOXES[box], storage=storage, tau=0.8, init_tg_amp=0.02)
    if force:
        p.update(body_force=(force, 0, -force), forcing="guo" if box % 2 else "paper")
    sims = [lb.Simulation(dict(p, streaming=s)) for s in ("pull", "aa")]
    for n in (1, 1, 1, 18):
        for sim in sims:
            sim.step(n)
        a, b = (sim.populations() for sim in sims)
        assert np.isfinite(a).all() and np.array_equal(a, b)
