"""Performance cases: the calls that users of the coupled LB / polymer-MD library make, with seeded
inputs, the bytes and operations that they cannot do without, and their results in 64 bits.

A pass is a few LB steps through the public entry points and the read-out that follows them: the
fluid (density and velocity, or the 19 populations) and the chain (positions and velocities).  The
chain is computed in 32 bits (positions as an unevaluated pair), so its read-out is kept as 32-bit
values, which is how a trajectory is stored.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_0710_1272_gb300 import lbmd as lb

DEFAULT = dict(
    kind="box", nx=32, ny=16, nz=16, wall=1, pore=3, y_walls=0, n_beads=0, storage="f32", streaming="pull",
    forcing="paper", coupling="trilinear", tau=1.0, gx=0.0, eps=1.0, kappa=0.0, kT_fluid=0.0, solvent=1,
    steps=1, read="fields", count=0, n_min=0, n_max=0, tune=0,
)


def listed():
    return [
        # one coupled step and its read-out: a monitored or interactively driven small translocation
        # (the small parity box of the tests); latency and launches are all it costs
        dict(name="small_step", nx=32, ny=16, nz=16, n_beads=20, steps=1),
        # production stretch of a mid-size translocation with the paper's own LJ strength and viscosity,
        # read out every 32 steps (the N = 100 box of the ragged ensemble)
        dict(name="mid_run", nx=64, ny=32, nz=32, pore=5, n_beads=100, eps=2e-3, tau=0.8, steps=32,
             read="populations"),
        # the headline translocation, single precision: 256 x 128 x 128, 5 x 5 pore, 400 beads
        dict(name="translocation_f32", nx=256, ny=128, nz=128, pore=5, n_beads=400, eps=2e-3, steps=16,
             read="populations"),
        # the same with 16-bit populations, the faster way to run it
        dict(name="translocation_f16", nx=256, ny=128, nz=128, pore=5, n_beads=400, eps=2e-3, steps=16,
             storage="f16", read="populations"),
        # the same with one population buffer, for boxes that fill the memory
        dict(name="translocation_aa", nx=256, ny=128, nz=128, pore=5, n_beads=400, eps=2e-3, steps=16,
             streaming="aa", read="populations"),
        # pure solvent with a body force (viscosity and decay-rate runs): the largest single box
        dict(name="solvent_f32", nx=256, ny=256, nz=256, wall=0, pore=0, gx=1e-6, steps=8),
        # Poiseuille channel of odd size with Guo forcing and bfloat16 populations, read as populations
        dict(name="channel_bf16", nx=255, ny=131, nz=127, wall=0, pore=0, y_walls=1, gx=1e-5, forcing="guo",
             storage="bf16", tau=0.8, steps=8, read="populations"),
        # fluctuating solvent (thermal source in every non-conserved mode)
        dict(name="thermal_f32", nx=128, ny=128, nz=128, wall=0, pore=0, kT_fluid=1e-4, tau=0.8, steps=8,
             read="populations"),
        # comparison run without a solvent: a long stiff chain, MD only
        dict(name="chain_free", nx=192, ny=96, nz=96, pore=5, n_beads=700, eps=2e-3, kappa=0.05, solvent=0,
             steps=16, read="none"),
        # translocation statistics: a ragged batch of long chains with 16-bit populations, launch shape
        # picked by the library's autotuner, as a statistics run does before its long loop
        dict(name="ensemble_f16", kind="ensemble", count=32, n_min=120, n_max=400, eps=2e-3, storage="f16", steps=32,
             tune=1),
        # a small batch of short chains in free solvent (gyration and diffusion averages), single
        # precision, the launch shape left at its default
        dict(name="ensemble_f32", kind="ensemble", count=16, n_min=20, n_max=100, wall=0, pore=0, eps=2e-3, steps=32),
        # one solvent step on the caller's own populations (no context, nothing allocated), walls and pore
        dict(name="noalloc_step", kind="noalloc", nx=160, ny=96, nz=96, pore=5, gx=1e-5, forcing="guo", tau=0.9),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _length(n):
    """Beads of a chain.  One more than a multiple of 32 is passed over: there the constraint solve has
    lost the chain's last bond in releases of the library, so no result exists to hold others against."""
    return int(n) + (n > 32 and n % 32 == 1)


def draw(rng):
    kind = rng.choice(["coupled", "coupled", "coupled", "solvent", "solvent", "thermal", "free", "ensemble",
                       "ensemble", "noalloc"])
    store = rng.choice(["f32", "f16", "bf16"])
    c = {}
    if kind == "coupled":
        n = _length(_log(rng, 2, 600))
        side = max(12, 2.2 * n ** 0.6)
        c.update(nx=int(side * rng.uniform(2.0, 3.0)), ny=int(side * rng.uniform(1.0, 1.6)),
                 nz=int(side * rng.uniform(1.0, 1.6)), pore=rng.choice([3, 4, 5]), n_beads=n,
                 storage=store, streaming=rng.choice(["pull", "pull", "aa"]), tau=rng.choice([0.7, 0.8, 1.0]),
                 eps=rng.choice([1.0, 2e-3]), kappa=rng.choice([0.0, 0.0, 0.02]),
                 coupling=rng.choice(["trilinear", "trilinear", "ngp"]), steps=rng.choice([1, 2, 5, 16, 24]),
                 read=rng.choice(["fields", "populations"]))
    elif kind in ("solvent", "thermal"):
        top = 5_000_000 if kind == "solvent" else 1_000_000
        v = math.exp(rng.uniform(math.log(3000), math.log(top)))
        a, b = rng.uniform(0.6, 1.6), rng.uniform(0.6, 1.6)
        side = v ** (1 / 3)
        wall, y_walls = rng.choice([(0, 0), (0, 0), (0, 1), (1, 0)])
        c.update(nx=max(8, int(side * a)), ny=max(8, int(side * b)), nz=max(8, int(side / (a * b))), wall=wall,
                 y_walls=y_walls, pore=3 if wall else 0, storage=store, streaming=rng.choice(["pull", "pull", "aa"]),
                 forcing=rng.choice(["paper", "guo"]), gx=rng.choice([0.0, 1e-5]), tau=rng.choice([0.7, 0.8, 1.0]),
                 kT_fluid=1e-4 if kind == "thermal" else 0.0, steps=rng.choice([1, 3, 8, 16]),
                 read=rng.choice(["fields", "populations"]))
    elif kind == "free":
        n = _length(_log(rng, 2, 1000))
        side = max(16, 2.2 * n ** 0.6)
        c.update(nx=int(2.2 * side), ny=int(1.2 * side), nz=int(1.2 * side), pore=5, n_beads=n, eps=2e-3,
                 kappa=rng.choice([0.0, 0.05]), solvent=0, steps=rng.choice([1, 8, 16, 32]), read="none")
    elif kind == "ensemble":
        # behind a wall only chains that take thousands of steps to cross it: a realisation ends there
        wall = rng.choice([0, 1])
        lo = _log(rng, 130, 170) if wall else _log(rng, 10, 60)
        c.update(kind="ensemble", count=rng.randint(3, 10 if wall else 24), n_min=lo,
                 n_max=int(lo * rng.uniform(1.0, 1.5 if wall else 4.0)), wall=wall, pore=3 if wall else 0,
                 storage=store, eps=2e-3, steps=rng.choice([4, 16, 32]), tune=rng.choice([0, 1]))
    else:
        v = math.exp(rng.uniform(math.log(3000), math.log(3_000_000)))
        a = rng.uniform(0.7, 1.5)
        side = v ** (1 / 3)
        wall, y_walls = rng.choice([(0, 0), (0, 1), (1, 0)])
        c.update(kind="noalloc", nx=max(12, int(side * a)), ny=max(12, int(side)), nz=max(12, int(side / a)),
                 wall=wall, y_walls=y_walls, pore=5 if wall else 0, gx=rng.choice([0.0, 1e-5]),
                 forcing=rng.choice(["paper", "guo"]), tau=rng.choice([0.7, 0.9, 1.0]))
    return c


# ---- inputs ------------------------------------------------------------------------------------
SIGMA, BOND, GAMMA, KT, DRIVE, SUBSTEPS = 1.8, 1.2, 0.1, 1e-4, 0.02, 5
RC = 2 ** (1 / 6) * SIGMA


def _geometry(c):
    """(first wall layer or -1, pore origin y, z) of a case."""
    return (c["nx"] // 2 if c["wall"] else -1), (c["ny"] - c["pore"]) // 2, (c["nz"] - c["pore"]) // 2


def _chain(c, rng):
    """Self-avoiding start on the cis side, its first bead in the pore mouth (mid-box without a wall)."""
    n, box = c["n_beads"], np.array([c["nx"], c["ny"], c["nz"]], dtype=np.float64)
    wx, y0, z0 = _geometry(c)
    mouth = np.array([wx + 1.0, y0 + (c["pore"] - 1) / 2, z0 + (c["pore"] - 1) / 2]) if wx >= 0 else box / 2
    pos = np.zeros((n, 3))
    pos[0] = mouth
    if n > 1:
        pos[1] = mouth + [BOND, 0, 0]
    i, failed = 2, 0
    while i < n:
        step = rng.normal(size=(12, 3))
        trial = pos[i - 1] + BOND * step / np.linalg.norm(step, axis=1, keepdims=True)
        ok = np.ones(12, dtype=bool)
        if wx >= 0:
            ok = (trial[:, 0] >= wx + RC) & (trial[:, 0] <= wx + box[0] - RC)
        d = trial[:, None, :] - pos[None, : i - 1]
        d -= box * np.rint(d / box)
        ok &= (np.einsum("ijk,ijk->ij", d, d) >= RC * RC).all(axis=1)
        if ok.any():
            pos[i] = trial[np.argmax(ok)]
            i += 1
        else:
            failed += 1
            if failed % 8 == 0:  # a dead end
                i = max(2, i - 12)
    return pos


def _member(c, seed):
    """Library parameters of a box case and its chain start."""
    rng = np.random.default_rng([17, int(seed)])
    wx, _, _ = _geometry(c)
    p = dict(nx=c["nx"], ny=c["ny"], nz=c["nz"], wall_x=wx, pore_d=c["pore"] if wx >= 0 else 0, y_walls=c["y_walls"],
             storage=c["storage"], streaming=c["streaming"], forcing=c["forcing"], coupling=c["coupling"],
             n_beads=c["n_beads"], md_substeps=SUBSTEPS, tau=c["tau"], body_force=(c["gx"], 0.0, 0.0), gamma=GAMMA,
             kT=KT, lj_sigma=SIGMA, lj_eps=c["eps"], kappa_phi=c["kappa"], f_drive=DRIVE, bond_len=BOND,
             kT_fluid=c["kT_fluid"], hydrodynamics=c["solvent"], seed=int(rng.integers(1, 1 << 40)),
             init_tg_amp=float(np.float32(rng.uniform(0.01, 0.02))))
    return p, (_chain(c, rng) if c["n_beads"] else None)


def _member_cases(c):
    """Box cases of an ensemble: lengths spread over [n_min, n_max], boxes that grow with the chain."""
    got = []
    for k in range(c["count"]):
        n = _length(round(c["n_min"] * (c["n_max"] / c["n_min"]) ** (k / max(1, c["count"] - 1))))
        side = [max(16 * low, int(a * n ** 0.6 / 16 + 0.5) * 16) for a, low in ((4, 2), (2, 1), (2, 1))]
        got.append(dict(c, kind="box", n_beads=n, nx=side[0], ny=side[1], nz=side[2],
                        pore=(3, 5)[k % 2] if c["wall"] else 0))
    return got


def _members(c, seed):
    """The realisations of an ensemble: box case, library parameters and chain start of each."""
    rng = np.random.default_rng([29, int(seed)])
    return [(m, *_member(m, int(rng.integers(1 << 30)))) for m in _member_cases(c)]


def _caller_populations(c, seed):
    """Pre-collision populations f_p of a mildly perturbed fluid, as a caller of the bare step holds them."""
    g = torch.Generator(device=_device())
    g.manual_seed(int(seed) + 1000)
    w = torch.tensor(W, dtype=torch.float32, device=_device())
    noise = torch.rand((19, c["nz"], c["ny"], c["nx"]), generator=g, device=_device(), dtype=torch.float32)
    return w[:, None, None, None] * (1.0 + 0.1 * (noise - 0.5))


def _device():
    return "cuda" if torch.cuda.is_available() else "cpu"


def prepare(case, seed):
    c = dict(DEFAULT, **case)
    if c["kind"] == "ensemble":
        got = _members(c, seed)
        ens = lb.Ensemble([p for _, p, _ in got], [pos for _, _, pos in got])
        if c["tune"]:
            ens.autotune(2)
        return dict(c=c, ens=ens, shapes=[(m["nz"], m["ny"], m["nx"]) for m, _, _ in got])
    if c["kind"] == "noalloc":
        p, _ = _member(c, seed)
        params, keep = lb.make_params(p)
        f = _caller_populations(c, seed)
        return dict(c=c, params=params, keep=keep, f=f, out=torch.empty_like(f))
    p, pos = _member(c, seed)
    return dict(c=c, sim=lb.Simulation(p, init_pos=pos))


def _beads(n):
    return torch.empty((2, n, 3), dtype=torch.float64, device="cuda")


def run(state):
    c = state["c"]
    if c["kind"] == "noalloc":
        lb.lbmd_lb_step_noalloc(state["params"], state["f"].data_ptr(), state["out"].data_ptr(),
                                torch.cuda.current_stream().cuda_stream)
        return {"f": state["out"]}
    if c["kind"] == "ensemble":
        ens = state["ens"]
        ens.step(c["steps"])
        r = ens.results()
        beads = _beads(sum(ens.N))
        flat = torch.empty(sum(19 * a * b * d for a, b, d in state["shapes"]), dtype=torch.float32, device="cuda")
        i = o = 0
        for k, n in enumerate(ens.N):
            lb.lbmd_ensemble_read_beads(ens.ens, k, beads[0, i:].data_ptr(), beads[1, i:].data_ptr(), 1)
            lb.lbmd_ensemble_read_populations(ens.ens, k, flat[o:].data_ptr(), 1)
            i, o = i + n, o + 19 * math.prod(state["shapes"][k])
        chain = beads.float()
        return {"pos": chain[0], "vel": chain[1], "f": flat, "state": r["state"], "steps": r["steps"]}
    sim = state["sim"]
    sim.step(c["steps"])
    out = {}
    if c["read"] == "fields":
        out["rho"], out["u"] = sim.fields_device()
    elif c["read"] == "populations":
        out["f"] = sim.populations_device()
    if c["n_beads"]:
        beads = _beads(c["n_beads"])
        lb.lbmd_read_beads(sim.ctx, beads[0].data_ptr(), beads[1].data_ptr(), 1)
        chain = beads.float()
        out["pos"], out["vel"] = chain[0], chain[1]
    return out


# ---- what a pass cannot do without ---------------------------------------------------------------
def _solid_count(c):
    wx, _, _ = _geometry(c)
    solid = (c["ny"] * c["nz"] - c["pore"] ** 2) if wx >= 0 else 0
    return solid + (2 * (c["nx"] - (1 if wx >= 0 else 0)) * c["nz"] if c["y_walls"] else 0)


def _box_work(c):
    nodes = c["nx"] * c["ny"] * c["nz"]
    fluid = nodes - _solid_count(c)
    held = 4 if c["storage"] == "f32" else 2
    bytes_, flops = 0.0, 0.0
    if c["solvent"]:
        # every step reads and writes the 19 populations of each fluid node once; about 260 operations
        # a node (moments, equilibrium, relaxation), 700 more for the fifteen normals and their modes
        bytes_ += c["steps"] * fluid * 2 * 19 * held
        flops += c["steps"] * fluid * (260 + (700 if c["kT_fluid"] else 0))
        if c["read"] != "none":
            bytes_ += fluid * 19 * held + nodes * (16 if c["read"] == "fields" else 76)
    # the chain: its state in and out once, a few hundred operations a bead and substep
    bytes_ += c["n_beads"] * 48
    flops += c["steps"] * SUBSTEPS * c["n_beads"] * 800
    return bytes_, flops


def work(case):
    c = dict(DEFAULT, **case)
    if c["kind"] == "ensemble":
        both = [_box_work(dict(m, read="populations")) for m in _member_cases(c)]
        return {"bytes": sum(b for b, _ in both), "flops": sum(f for _, f in both)}
    if c["kind"] == "noalloc":
        nodes = c["nx"] * c["ny"] * c["nz"]
        fluid = nodes - _solid_count(c)
        return {"bytes": 76.0 * (fluid + nodes), "flops": 260.0 * fluid}
    b, f = _box_work(c)
    return {"bytes": float(b), "flops": float(f)}


# ---- the same in 64 bits, from the equations alone -----------------------------------------------
C = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1), (1, 1, 0), (-1, -1, 0),
     (1, -1, 0), (-1, 1, 0), (1, 0, 1), (-1, 0, -1), (1, 0, -1), (-1, 0, 1), (0, 1, 1), (0, -1, -1), (0, 1, -1),
     (0, -1, 1)]
W = [1 / 3] + 6 * [1 / 18] + 12 * [1 / 36]
OPP = [0] + [p + 1 if p % 2 else p - 1 for p in range(1, 19)]


def _solid(c):
    s = torch.zeros((c["nz"], c["ny"], c["nx"]), dtype=torch.bool, device=_device())
    wx, y0, z0 = _geometry(c)
    if wx >= 0:
        s[:, :, wx] = True
        s[z0:z0 + c["pore"], y0:y0 + c["pore"], wx] = False
    if c["y_walls"]:
        s[:, 0] = s[:, -1] = True
    return s


def _philox(c0, c1, c2, c3, seed):
    """Philox4x32-10 on int64 tensors or arrays of 32-bit values."""
    m = 0xFFFFFFFF

    def mul(a, x):  # 32 x 32 -> (high, low), through 16-bit halves to stay within 63 bits
        lo, hi = a * (x & 0xFFFF), a * (x >> 16)
        mid = hi + (lo >> 16)
        return (mid >> 16) & m, ((mid << 16) | (lo & 0xFFFF)) & m
    k0, k1 = seed & m, (seed >> 32) & m
    for r in range(10):
        if r:
            k0, k1 = (k0 + 0x9E3779B9) & m, (k1 + 0xBB67AE85) & m
        h0, l0 = mul(0xD2511F53, c0)
        h1, l1 = mul(0xCD9E8D57, c2)
        c0, c1, c2, c3 = h1 ^ c1 ^ k0, l1, h0 ^ c3 ^ k1, l0
    return c0, c1, c2, c3


def _modes():
    e = np.zeros((19, 19))
    for p, (x, y, z) in enumerate(C):
        s = x * x + y * y + z * z
        e[:, p] = [1, x, y, z, s - 1, 3 * x * x - s, y * y - z * z, x * y, y * z, z * x, (3 * s - 5) * x,
                   (3 * s - 5) * y, (3 * s - 5) * z, (y * y - z * z) * x, (z * z - x * x) * y, (x * x - y * y) * z,
                   3 * s * s - 6 * s + 1, (2 * s - 3) * (3 * x * x - s), (2 * s - 3) * (y * y - z * z)]
    return e


class _Fluid:
    """D3Q19 BGK on pre-collision populations f (Eqs. 5-8), halfway bounce-back, pull streaming."""

    def __init__(self, c, p, f=None):
        self.c, self.p, self.solid = c, p, _solid(c)
        self.g = torch.tensor(p["body_force"], dtype=torch.float64, device=_device())
        self.from_solid = [torch.roll(self.solid, (z, y, x), (0, 1, 2)) for x, y, z in C]
        if f is None:
            dev = dict(dtype=torch.float64, device=_device())
            x = 2 * math.pi * torch.arange(c["nx"], **dev) / c["nx"]
            y = 2 * math.pi * torch.arange(c["ny"], **dev)[:, None] / c["ny"]
            u = torch.zeros((3, c["nz"], c["ny"], c["nx"]), **dev)
            u[0] = p["init_tg_amp"] * torch.sin(x) * torch.cos(y)
            u[1] = -p["init_tg_amp"] * torch.cos(x) * torch.sin(y)
            f = self.equilibrium(torch.ones_like(u[0]), u)
        self.f = f
        self.f[:, self.solid] = 0

    def equilibrium(self, rho, u):
        sq = 1.5 * (u * u).sum(0)
        f = torch.empty((19,) + tuple(rho.shape), dtype=torch.float64, device=rho.device)
        for p, (x, y, z) in enumerate(C):
            cu = x * u[0] + y * u[1] + z * u[2]
            f[p] = W[p] * rho * (1 + 3 * cu + 4.5 * cu * cu - sq)
        return f

    def moments(self):
        rho = self.f.sum(0)
        j = torch.stack([sum(C[p][a] * self.f[p] for p in range(1, 19) if C[p][a]) for a in range(3)])
        if self.c["forcing"] == "guo":
            j = j + 0.5 * self.g[:, None, None, None]
        safe = torch.where(self.solid, torch.ones_like(rho), rho)
        return torch.where(self.solid, torch.zeros_like(rho), rho), torch.where(self.solid, torch.zeros_like(j), j / safe)

    def noise(self, rho, step):
        node = torch.arange(rho.numel(), dtype=torch.int64, device=rho.device).reshape(rho.shape)
        e, damp = _modes(), 1 - 1 / self.p["tau"]
        norms = []
        for block in range(4):
            x = _philox(node, torch.full_like(node, step), torch.zeros_like(node),
                        torch.full_like(node, block | 2 << 8), self.p["seed"])
            u = [((v >> 9).double() + 0.5) * 2.0 ** -23 for v in x]
            for a, b in ((u[0], u[1]), (u[2], u[3])):
                r = torch.sqrt(-2 * torch.log(a))
                norms += [r * torch.cos(2 * math.pi * b), r * torch.sin(2 * math.pi * b)]
        xi = torch.zeros_like(self.f)
        for k in range(4, 19):
            bk = sum(W[p] * e[k, p] ** 2 for p in range(19))
            t = math.sqrt(3 * self.p["kT_fluid"] * (1 - damp * damp) / bk) * torch.sqrt(rho) * norms[k - 4]
            for p in range(19):
                if e[k, p]:
                    xi[p] += W[p] * e[k, p] * t
        return xi

    def step(self, step, force=None):
        """One stream-collide; `force`: (flat nodes, forces) of the chain's reaction."""
        rho, u = self.moments()
        w = 1 / self.p["tau"]
        feq = self.equilibrium(rho, u)
        post = self.f + w * (feq - self.f)
        del feq
        gu = (self.g[:, None, None, None] * u).sum(0)
        for p, (x, y, z) in enumerate(C):
            cg = x * self.g[0] + y * self.g[1] + z * self.g[2]
            if self.c["forcing"] == "guo":
                cu = x * u[0] + y * u[1] + z * u[2]
                post[p] += (1 - 0.5 * w) * W[p] * (3 * (cg - gu) + 9 * cu * cg)
            else:
                post[p] += 3 * W[p] * cg
        if self.p["kT_fluid"] > 0:
            post += self.noise(rho, step)
        if force is not None:
            at, value = (torch.from_numpy(np.ascontiguousarray(v)).to(post.device) for v in force)
            for p in range(1, 19):
                c = torch.tensor(C[p], dtype=torch.float64, device=post.device)
                post[p].view(-1).index_add_(0, at, 3 * W[p] * (value @ c))
        new = torch.empty_like(post)
        for p, (x, y, z) in enumerate(C):
            new[p] = torch.where(self.from_solid[p], post[OPP[p]], torch.roll(post[p], (z, y, x), (0, 1, 2)))
        new[:, self.solid] = 0
        self.f = new


def _tridiagonal(sub, diag, sup, rhs):
    a = np.zeros((len(diag), len(diag)))
    i = np.arange(len(diag))
    a[i, i], a[i[1:], i[:-1]], a[i[:-1], i[1:]] = diag, sub[1:], sup[:-1]
    return np.linalg.solve(a, rhs)


class _Chain:
    """The M substeps of Sec. II: WCA, bending, walls, drive, drag, noise, SHAKE and RATTLE."""

    def __init__(self, c, p, pos):
        self.c, self.p, self.r, self.v = c, p, pos.copy(), np.zeros_like(pos)
        self.box = np.array([c["nx"], c["ny"], c["nz"]], dtype=np.float64)
        self.n = len(pos)
        self.solid = _solid(c).cpu().numpy()

    def wca(self, d):
        r2 = (d * d).sum(-1)
        near = (r2 < RC * RC) & (r2 > 0)
        s6 = np.where(near, SIGMA ** 2 / np.where(near, r2, 1), 0) ** 3
        return (24 * self.p["lj_eps"] * (2 * s6 * s6 - s6) / np.where(near, r2, 1))[..., None] * d

    def forces(self):
        n, r = self.n, self.r
        d = r[:, None] - r[None]
        d -= self.box * np.rint(d / self.box)
        i = np.arange(n)
        d[np.abs(i[:, None] - i[None]) <= 1] = 1e9
        f = self.wca(d).sum(1)
        wx, y0, z0 = _geometry(self.c)
        if wx >= 0 or self.c["y_walls"]:
            o = np.stack(np.meshgrid(*3 * [np.arange(-2, 4)], indexing="ij"), -1).reshape(-1, 3)
            node = np.floor(r)[:, None].astype(np.int64) + o
            x, y, z = np.moveaxis(node % self.box.astype(np.int64), -1, 0)
            w = np.where(self.solid[z, y, x][..., None], r[:, None] - node, 1e9)
            f += self.wca(w).sum(1)
        if wx >= 0 and self.c["pore"]:
            q = np.mod(r, self.box)
            dx = np.mod(r[:, 0] - wx + self.box[0] / 2, self.box[0]) - self.box[0] / 2
            d5 = self.c["pore"] - 0.5
            f[:, 0] -= DRIVE * ((np.abs(dx) <= 1.5) & (q[:, 1] >= y0 - 0.5) & (q[:, 1] < y0 + d5)
                                & (q[:, 2] >= z0 - 0.5) & (q[:, 2] < z0 + d5))
        if self.p["kappa_phi"] and n > 2:
            b = np.diff(r, axis=0)
            b1, b2 = b[:-1], b[1:]
            l1, l2 = np.linalg.norm(b1, axis=1)[:, None], np.linalg.norm(b2, axis=1)[:, None]
            cos = np.clip((b1 * b2).sum(1)[:, None] / (l1 * l2), -1, 1)
            phi = np.arccos(cos)
            a = self.p["kappa_phi"] * np.where(phi < 1e-4, 1, phi / np.where(phi < 1e-4, 1, np.sin(phi)))
            g1, g2 = b2 / (l1 * l2) - cos * b1 / l1 ** 2, b1 / (l1 * l2) - cos * b2 / l2 ** 2
            f[:-2] -= a * g1
            f[1:-1] += a * (g1 - g2)
            f[2:] += a * g2
        return f

    def noise(self, step, k):
        z = np.zeros(self.n, dtype=np.int64)
        x = _philox(np.arange(self.n, dtype=np.int64), z + step, z, z + k, self.p["seed"])
        u = [((v >> 9) + 0.5) * 2.0 ** -23 for v in x]
        a, b = np.sqrt(-2 * np.log(u[0])), np.sqrt(-2 * np.log(u[2]))
        return np.stack([a * np.cos(2 * np.pi * u[1]), a * np.sin(2 * np.pi * u[1]), b * np.cos(2 * np.pi * u[3])], 1)

    def cycle(self, step, ui):
        """M substeps with the fluid velocity frozen; returns the impulse handed over."""
        dt, j = 1 / SUBSTEPS, np.zeros_like(self.r)
        for k in range(SUBSTEPS):
            give = -GAMMA * (self.v - ui) + math.sqrt(2 * GAMMA * KT / dt) * self.noise(step, k)
            self.v = self.v + dt * (self.forces() + give)
            j += dt * give
            move = dt * self.v
            if self.n > 1:
                s = np.diff(self.r, axis=0)
                pad = np.zeros((1, 3))
                for _ in range(30):
                    d = s + np.diff(move, axis=0)
                    gap = (d * d).sum(1) - BOND ** 2
                    if np.abs(gap).max() < 1e-14:
                        break
                    sub, sup = np.zeros(self.n - 1), np.zeros(self.n - 1)
                    sub[1:], sup[:-1] = 2 * (d[1:] * s[:-1]).sum(1), 2 * (d[:-1] * s[1:]).sum(1)
                    x = _tridiagonal(sub, -4 * (d * s).sum(1), sup, -gap)[:, None] * s
                    move = move + np.concatenate([x, pad]) - np.concatenate([pad, x])
                self.v = move / dt
                d = s + np.diff(move, axis=0)
                sub, sup = np.zeros(self.n - 1), np.zeros(self.n - 1)
                sub[1:] = sup[:-1] = (d[1:] * d[:-1]).sum(1)
                x = _tridiagonal(sub, -2 * (d * d).sum(1), sup, -(d * np.diff(self.v, axis=0)).sum(1))[:, None] * d
                self.r = self.r + move
                self.v = self.v + np.concatenate([x, pad]) - np.concatenate([pad, x])
            else:
                self.r = self.r + move
        return j

    def corners(self):
        """(flat node, weight) of the transfer nodes of every bead."""
        cell = np.floor(self.r).astype(np.int64)
        s = self.r - cell
        o = np.array([[k & 1, k >> 1 & 1, k >> 2 & 1] for k in range(8)])
        if self.c["coupling"] == "ngp":
            node, w = (cell + (s >= 0.5))[:, None], np.ones((self.n, 1))
        else:
            node = cell[:, None] + o
            w = np.where(o[None], s[:, None], 1 - s[:, None]).prod(-1)
        x, y, z = np.moveaxis(node % self.box.astype(np.int64), -1, 0)
        w = np.where(self.solid[z, y, x], 0, w)
        total = w.sum(1, keepdims=True)
        return (z * self.c["ny"] + y) * self.c["nx"] + x, w / np.where(total > 0, total, 1)


def _advance(c, p, pos, steps):
    fluid = _Fluid(c, p) if c["solvent"] else None
    chain = _Chain(c, p, pos) if c["n_beads"] else None
    for t in range(steps):
        force = None
        if chain is not None:
            ui = np.zeros((chain.n, 3))
            if fluid is not None:
                at, w = chain.corners()
                u = fluid.moments()[1].reshape(3, -1)[:, torch.from_numpy(at).to(_device())].cpu().numpy()
                ui = np.einsum("aik,ik->ia", u, w)
            j = chain.cycle(t, ui)
            if fluid is not None:
                force = at.reshape(-1), (-w[:, :, None] * j[:, None]).reshape(-1, 3)
        if fluid is not None:
            fluid.step(t, force)
    return fluid, chain


def exact(case, seed):
    c = dict(DEFAULT, **case)
    if c["kind"] == "noalloc":
        p, _ = _member(c, seed)
        fluid = _Fluid(c, p, _caller_populations(c, seed).double())
        fluid.step(0)
        return {"f": fluid.f}
    if c["kind"] == "ensemble":
        got = _members(c, seed)
        if sum(len(pos) for _, _, pos in got) * c["steps"] > 30_000:
            return None  # too many chains for plain numpy
        done = [_advance(m, p, pos, c["steps"]) for m, p, pos in got]
        return {"pos": np.concatenate([chain.r for _, chain in done]),
                "vel": np.concatenate([chain.v for _, chain in done]),
                "f": torch.cat([fluid.f.reshape(-1) for fluid, _ in done]), "state": None, "steps": None}
    p, pos = _member(c, seed)
    fluid, chain = _advance(c, p, pos, c["steps"])
    out = {}
    if c["read"] == "fields":
        out["rho"], out["u"] = fluid.moments()
    elif c["read"] == "populations":
        out["f"] = fluid.f
    if chain is not None:
        out["pos"], out["vel"] = chain.r, chain.v
    return out
