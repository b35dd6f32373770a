"""Bead states and velocity fields of runs whose last bits matter: chains of stiff beads, and chains in
16-bit populations, carry a different last bit of the MD cycle into the fifth digit of the velocities
within twenty steps, and thermal noise rounded to 16 bits does the same to the field, so a change of their
arithmetic shows here and nowhere else.  The values in
golden/*.npz were written by ``python tests/released_values.py KIND golden/KIND_values.npz`` with the
release of commit 33770b1 (CUDA 13.0); the tests compare the present library with them."""
import os
import sys

import numpy as np

HERE = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, os.path.dirname(HERE))

_CHAIN = dict(wall_thickness=1, gamma=0.1, kT=1e-4, lj_sigma=1.8, f_drive=0.02, bond_len=1.2, md_substeps=5,
              init_tg_amp=0.015)
CASES = {
    "chain": {
        "f32_130": (dict(nx=84, ny=44, nz=58, wall_x=42, pore_d=5, n_beads=130, lj_eps=1.0, seed=29), 16),
        "f32_266": (dict(nx=144, ny=76, nz=84, wall_x=72, pore_d=3, n_beads=266, lj_eps=1.0, seed=20, tau=0.8), 16),
        "bf16_46": (dict(nx=46, ny=22, nz=22, wall_x=23, pore_d=4, n_beads=46, lj_eps=1.0, kappa_phi=0.02, seed=6,
                         storage="bf16"), 16),
        "bf16_aa_9": (dict(nx=32, ny=13, nz=14, wall_x=16, pore_d=3, n_beads=9, lj_eps=1.0, seed=23, tau=0.7,
                           storage="bf16", streaming="aa"), 24),
        "f16_100": (dict(nx=64, ny=32, nz=32, wall_x=32, pore_d=5, n_beads=100, lj_eps=1.0, kappa_phi=0.02, seed=4,
                         storage="f16"), 24),
        "bf16_300": (dict(nx=128, ny=64, nz=64, wall_x=64, pore_d=5, n_beads=300, lj_eps=1.0, seed=8,
                          storage="bf16"), 12),
    },
    "thermal": {
        "bf16_pull": (dict(nx=26, ny=17, nz=12, kT_fluid=1e-4, tau=0.8, seed=3, storage="bf16"), 16),
        "bf16_aa_guo": (dict(nx=24, ny=19, nz=14, kT_fluid=1e-4, tau=0.7, seed=4, storage="bf16", streaming="aa",
                             forcing="guo", body_force=(1e-5, 0.0, 0.0)), 16),
        "f16_walls": (dict(nx=27, ny=18, nz=15, wall_x=13, pore_d=3, kT_fluid=1e-4, seed=5, storage="f16",
                           body_force=(1e-5, 0.0, 0.0)), 16),
        "f16_above_2^15": (dict(nx=41, ny=33, nz=27, y_walls=1, kT_fluid=1e-4, tau=0.8, seed=6, storage="f16"), 9),
        "f32": (dict(nx=25, ny=18, nz=13, kT_fluid=1e-4, tau=0.8, seed=7), 16),
        "f32_chain": (dict(nx=84, ny=44, nz=58, wall_x=42, pore_d=5, n_beads=130, lj_eps=1.0, kT_fluid=1e-4,
                           seed=29), 16),
        "bf16_chain": (dict(nx=34, ny=16, nz=16, wall_x=17, pore_d=3, n_beads=24, lj_eps=1.0, kT_fluid=1e-4, seed=9,
                            storage="bf16", streaming="aa"), 16),
    },
}


def run(kind, name):
    """{array name: float32 array} of a case after its steps; the velocity field at every 7th node."""
    import paper_0710_1272_gb300 as lb

    p, steps = CASES[kind][name]
    sim = lb.Simulation(dict(_CHAIN, **p))
    sim.step(steps)
    out = {}
    if p.get("n_beads", 0):
        pos, vel = sim.beads()
        out["pos"], out["vel"] = pos.astype(np.float32), vel.astype(np.float32)
    if p["nx"] * p["ny"] * p["nz"] < 40000:
        rho, u = sim.fields()
        out["rho"], out["u"] = rho.reshape(-1)[::7].copy(), u.reshape(3, -1)[:, ::7].copy()
    return out


def golden(kind):
    return np.load(os.path.join(HERE, "golden", kind + "_values.npz"))


def distance(got, want):
    """2-norm of the difference over that of the released values."""
    a, b = got.astype(np.float64), want.astype(np.float64)
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


if __name__ == "__main__":
    kind, path = sys.argv[1:3]
    np.savez_compressed(path, **{n + "." + k: v for n in CASES[kind] for k, v in run(kind, n).items()})
