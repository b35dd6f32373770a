"""16-bit storage by pairs of nodes, in place and pull: the same bits after every step,
widths even and odd, walls at either half of a word, the box's edges and the pore
included.  Pull streaming takes pairs above 2^15 nodes, the in-place odd step from 2^17
(with a wall across x from 192 nodes in x), so the boxes between hold pairs against
single nodes."""
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
    dict(nx=191, ny=31, nz=24, wall_x=100, pore_d=5),                     # odd step by single nodes
    dict(nx=33, ny=32, nz=33, wall_x=16, pore_d=5),
    dict(nx=35, ny=31, nz=31, wall_x=34, pore_d=3),
    dict(nx=37, ny=30, nz=31, y_walls=1),
    dict(nx=34, ny=32, nz=32, wall_x=33, wall_thickness=2, pore_d=4),
    dict(nx=32, ny=32, nz=32, wall_x=15, pore_d=3),                       # 2^15: pull by single nodes
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
