"""The work that a user of this framework has it do, as cases that can be timed and compared.

A case is a dict of plain values.  ``listed()`` names the standing ones, ``draw(rng)`` gives more of
the same ranges, ``prepare(case, seed)`` makes what a program has in hand before the call (initial
states on the GPU and the system that holds them), ``run(state)`` is one pass through the public
entry points, ``work(case)`` what the pass cannot do without, and ``exact(case, seed)`` the same
outputs in 64 bits from plain torch operations.

Systems with FP32 pair forces write their frames, forces, gradients and rows of measured quantities
in FP32, as trajectory files do; MD_FP64 systems keep FP64.
"""
import ctypes
import itertools
import math

import numpy as np
import torch

from paper_2003_14061_gb300 import binding
from paper_2003_14061_gb300.system import MDSystem, make_params

WCA = 2.0 ** (1.0 / 6.0)
DT = 0.005
CHAIN = {"length": 25, "fene_k": 30.0, "fene_r0": 1.5, "bend_k": 3.0, "dihedral_k": 0.0}
NLAG, ORIGIN_EVERY = 50, 10          # VACF / MSD: lags followed, samples between time origins


# ---------------------------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------------------------
def _fluid(name, cells, n, lj, **kw):
    """A soft-sphere (WCA) fluid or a Lennard-Jones liquid of n atoms on nx x ny x nz fcc cells."""
    nx, ny, nz = cells
    c = {"name": name} if name else {}
    c.update({"kind": "run", "nx": nx, "ny": ny, "nz": nz, "n": n, "steps": 20, "precision": "mixed",
              "rule": "vmax", "props_every": 0})
    c.update({"rho": 0.8442, "temp": 0.72, "rc": 2.5, "skin": 0.3} if lj else
             {"rho": 0.8, "temp": 1.0, "rc": WCA, "skin": 0.4})
    c.update(kw)
    return c


def listed():
    return [
        # forces of a small configuration from inside another program's step, nothing allocated: the
        # smallest call there is, bound by its launches
        _fluid("static_forces_5k", (11, 11, 11), 5003, False, kind="static", steps=1),
        # a small validation run in FP64 on a plain cell list rebuilt at every step
        _fluid("cell_list_2k_fp64", (8, 8, 8), 2048, False, precision="fp64", rule="every", skin=0.0, steps=100),
        # a small liquid, its energy, pressure and momentum logged every 10 steps
        _fluid("lj_4k_log10", (10, 10, 10), 4000, True, props_every=10, steps=100),
        # FP32 state, a ragged number of atoms in a long box, the exact-displacement rebuild rule
        _fluid("wca_100k_fp32", (24, 30, 38), 100003, False, precision="fp32", rule="disp", steps=50),
        # the usual size of a production liquid
        _fluid("lj_256k", (40, 40, 40), 256000, True, steps=50),
        # an outer program (sampler, minimiser, checkpoint restart) hands over new positions and
        # wants their forces: upload, binning, neighbour matrix, one force pass
        _fluid("new_positions_500k", (50, 50, 50), 500000, True, kind="forces", steps=1),
        # velocity autocorrelation and diffusion of the dense soft-sphere fluid, sampled every 10 steps
        {"name": "diffusion_1m", "kind": "dynamics", "nx": 100, "ny": 100, "nz": 100, "n": 1000000, "rho": 1.0,
         "temp": 1.0, "rc": WCA, "skin": 0.4, "steps": 10, "samples": 5, "precision": "mixed", "rule": "vmax",
         "props_every": 0},
        # gradients of a trajectory loss: forward, recompute and reverse
        _fluid("adjoint_32k", (20, 20, 20), 32000, False, kind="adjoint", steps=40, ckpt=10),
        # uneven polymer melts side by side (chains of 25 beads)
        {"name": "chains_64", "kind": "chains", "nrep": 64, "emin": 10, "emax": 17, "rho": 0.85, "temp": 1.0,
         "rc": WCA, "skin": 0.4, "steps": 50, "precision": "mixed", "rule": "vmax", "props_every": 0},
        # hundreds of uneven independent systems advanced together
        {"name": "batch_512", "kind": "batch", "nrep": 512, "nmin": 500, "nmax": 32000, "rhomin": 0.6, "rhomax": 0.9,
         "temp": 1.0, "rc": WCA, "skin": 0.4, "steps": 20, "precision": "mixed", "rule": "vmax", "props_every": 0},
        # the large fluid with every quantity measured at every step
        _fluid("wca_4m_log1", (100, 100, 100), 4000000, False, props_every=1, steps=20),
        # the largest liquid
        _fluid("lj_16m", (160, 160, 160), 16384000, True, steps=40),
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _cells_for(rng, n):
    """fcc cells of a box of up to 1 : 1.6 sides that hold at least n atoms."""
    m = (n / 4.0) ** (1.0 / 3.0)
    nx = max(5, int(round(m * rng.uniform(0.8, 1.1))))
    ny = max(5, int(round(m * rng.uniform(0.9, 1.2))))
    nz = max(5, int(math.ceil(n / (4.0 * nx * ny))))
    return nx, ny, nz


def draw(rng):
    kind = rng.choice(["run", "run", "run", "run", "static", "forces", "dynamics", "adjoint", "chains", "batch"])
    if kind == "batch":
        nrep = _log_uniform(rng, 16, 512)
        nmax = rng.randint(4000, 32000)
        return {"kind": kind, "nrep": nrep, "nmin": rng.randint(500, 2000), "nmax": nmax, "rhomin": 0.6,
                "rhomax": round(rng.uniform(0.75, 0.9), 3), "temp": 1.0, "rc": WCA, "skin": rng.choice([0.3, 0.4]),
                "steps": rng.randint(15, 25), "precision": rng.choice(["mixed", "mixed", "fp32"]), "rule": "vmax",
                "props_every": rng.choice([0, 0, 5])}
    if kind == "chains":
        return {"kind": kind, "nrep": _log_uniform(rng, 4, 128), "emin": rng.randint(8, 12),
                "emax": rng.randint(13, 20), "rho": round(rng.uniform(0.8, 0.9), 3), "temp": 1.0, "rc": WCA,
                "skin": 0.4, "steps": rng.randint(30, 60), "precision": rng.choice(["mixed", "fp32"]), "rule": "vmax",
                "props_every": 0}
    if kind == "dynamics":
        e = rng.randint(12, 110)
        return {"kind": kind, "nx": e, "ny": e + rng.randint(0, 4), "nz": e, "n": 0, "rho": 1.0, "temp": 1.0,
                "rc": WCA, "skin": 0.4, "steps": rng.randint(5, 12), "samples": rng.randint(3, 6),
                "precision": "mixed", "rule": "vmax", "props_every": 0}
    lj = rng.random() < 0.5
    if kind == "static":
        n = _log_uniform(rng, 2000, 60000)
        return _fluid("", _cells_for(rng, n), n, lj, kind=kind, steps=1)
    if kind == "forces":
        n = _log_uniform(rng, 3000, 2000000)
        return _fluid("", _cells_for(rng, n), n, lj, kind=kind, steps=1,
                      precision=rng.choice(["mixed", "mixed", "fp32"]))
    if kind == "adjoint":
        n = _log_uniform(rng, 2000, 40000)
        return _fluid("", _cells_for(rng, n), n, False, kind=kind, steps=rng.randint(20, 50), ckpt=rng.randint(5, 15))
    prec = rng.choice(["mixed", "mixed", "mixed", "fp32", "fp32", "fp64"])
    n = _log_uniform(rng, 2000, {"mixed": 8000000, "fp32": 2000000, "fp64": 40000}[prec])
    c = _fluid("", _cells_for(rng, n), n, lj, precision=prec, props_every=rng.choice([0, 0, 1, 10]),
               rule=rng.choice(["vmax", "vmax", "disp"]),
               steps=rng.randint(15, 25) if n > 200000 else rng.randint(40, 100))
    if prec == "fp64":
        c.update(rule=rng.choice(["every", "vmax"]))
        c.update(skin=0.0 if c["rule"] == "every" else c["skin"])
    else:
        c["skin"] = round(c["skin"] * rng.uniform(0.8, 1.2), 3)
    return c


# ---------------------------------------------------------------------------------------------
# initial states, on the GPU, from the seed alone
# ---------------------------------------------------------------------------------------------
_BASIS = ((0.25, 0.25, 0.25), (0.75, 0.75, 0.25), (0.75, 0.25, 0.75), (0.25, 0.75, 0.75))


def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) * 7919 + 17)
    return g


def _maxwell(n, temp, g):
    v = torch.randn(n, 3, dtype=torch.float64, device="cuda", generator=g)
    v -= v.mean(0, keepdim=True)
    return v * torch.sqrt(temp * 3.0 * (n - 1) / (v * v).sum())


def _wrapped(x, box):
    x = torch.remainder(x, box)
    return torch.where(x >= box, torch.zeros_like(x), x)


def _fcc(nx, ny, nz, n, rho, amp, g):
    """n atoms on the sites of nx x ny x nz fcc cells (a random subset where n is smaller), each
    displaced by up to amp per coordinate: (x, box)."""
    sites = 4 * nx * ny * nz
    pick = (torch.arange(n, device="cuda") if n == sites else
            torch.randperm(sites, device="cuda", generator=g)[:n].sort().values)
    a = (n / (rho * nx * ny * nz)) ** (1.0 / 3.0)
    box = torch.tensor([nx * a, ny * a, nz * a], dtype=torch.float64, device="cuda")
    cell, b = pick // 4, pick % 4
    x = torch.stack([cell % nx, (cell // nx) % ny, cell // (nx * ny)], 1).to(torch.float64)
    x += torch.tensor(_BASIS, dtype=torch.float64, device="cuda")[b]
    x *= a
    x += (2.0 * torch.rand(n, 3, dtype=torch.float64, device="cuda", generator=g) - 1.0) * amp
    return _wrapped(x, box), box


def _cubic(nx, ny, nz, rho, amp, g, serpentine=False):
    """A simple cubic grid (x, box); serpentine: sites ordered along a path through nearest sites."""
    k = np.arange(nx * ny * nz)
    iz, p = k // (nx * ny), k % (nx * ny)
    if serpentine:                                   # odd planes walk the plane's path backwards
        p = np.where(iz % 2 == 0, p, nx * ny - 1 - p)
    iy, ix = p // nx, p % nx
    if serpentine:
        ix = np.where(iy % 2 == 0, ix, nx - 1 - ix)
    a = rho ** (-1.0 / 3.0)
    x = torch.from_numpy((np.stack([ix, iy, iz], 1) + 0.5) * a).cuda()
    box = torch.tensor([nx * a, ny * a, nz * a], dtype=torch.float64, device="cuda")
    x += (2.0 * torch.rand(x.shape[0], 3, dtype=torch.float64, device="cuda", generator=g) - 1.0) * amp
    return _wrapped(x, box), box


def _replica_sizes(c):
    """(atoms, density) of each replica of a batch, or edges of each chain melt: part of the case."""
    r = np.random.Generator(np.random.PCG64(c["nrep"]))
    if c["kind"] == "chains":
        return [int(e) for e in r.integers(c["emin"], c["emax"] + 1, size=c["nrep"])]
    return list(zip((int(k) for k in r.integers(c["nmin"], c["nmax"] + 1, size=c["nrep"])),
                    (float(q) for q in r.uniform(c["rhomin"], c["rhomax"], size=c["nrep"]))))


def _state(c, seed):
    """(x, v, n_rep, boxes): positions and velocities [n, 3] of all replicas, atoms and box of each."""
    g = _gen(seed)
    if c["kind"] == "batch":
        parts = []
        for n, rho in _replica_sizes(c):
            m = int(math.ceil((n / 4.0) ** (1.0 / 3.0) - 1e-9))
            parts.append((*_fcc(m, m, m, n, rho, 0.03, g), n))
    elif c["kind"] == "chains":
        parts = [(*_cubic(e, e, e, c["rho"], 0.02, g, serpentine=True), e ** 3) for e in _replica_sizes(c)]
    elif c["kind"] == "dynamics":
        parts = [(*_cubic(c["nx"], c["ny"], c["nz"], c["rho"], 0.05, g), c["nx"] * c["ny"] * c["nz"])]
    else:
        parts = [(*_fcc(c["nx"], c["ny"], c["nz"], c["n"], c["rho"], 0.08, g), c["n"])]
    v = torch.cat([_maxwell(n, c["temp"], g) for _, _, n in parts])
    x = torch.cat([p[0] for p in parts])
    return x, v, [p[2] for p in parts], torch.stack([p[1] for p in parts])


# ---------------------------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------------------------
def prepare(case, seed):
    c = dict(case)
    x, v, n_rep, boxes = _state(c, seed)
    st = {"case": c, "x": x, "v": v, "f": None, "out_x": torch.empty_like(x), "out_v": torch.empty_like(v)}
    if c["kind"] == "static":
        st["params"] = make_params(rc=c["rc"], skin=0.0, n=c["n"], box=boxes[0].tolist())
        st["f"] = torch.empty_like(x)
        st["u"] = torch.empty(c["n"], dtype=torch.float64, device="cuda")
        binding.lib()
        return st
    geo = ({"n_rep": n_rep, "boxes": boxes.cpu().numpy()} if c["kind"] in ("batch", "chains") else
           {"box": boxes[0].cpu().numpy()})
    st["system"] = MDSystem(x, v, rc=c["rc"], skin=c["skin"], dt=DT, precision=c["precision"],
                            rebuild_rule=c["rule"], props_every=c["props_every"], **geo)
    if c["kind"] == "chains":
        st["system"].set_chains(**CHAIN)
    if c["kind"] == "dynamics":
        st["system"].dyn_begin(NLAG, ORIGIN_EVERY)
    if c["kind"] == "forces":
        # the positions that the outer program will ask about: those of another draw
        st["x"], st["v"], _, _ = _state(c, int(seed) + 500009)
        st["f"] = torch.empty_like(x)
    return st


def _frame(st):
    """The state as a program stores it: FP64 from MD_FP64 systems, FP32 from the others."""
    st["system"].state_into(st["out_x"], st["out_v"])
    if st["case"]["precision"] == "fp64":
        return {"x": st["out_x"], "v": st["out_v"]}
    return {"x": st["out_x"].float(), "v": st["out_v"].float()}


def run(st):
    c = st["case"]
    if c["kind"] == "static":
        ptr = [ctypes.c_void_p(t.data_ptr()) for t in (st["x"], st["f"], st["u"])]
        binding.call("md_forces_static", ctypes.byref(st["params"]), c["n"], *ptr,
                     ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
        return {"f": st["f"].float(), "u": st["u"].float()}
    s = st["system"]
    if c["kind"] == "forces":
        s.set_state(st["x"], st["v"])
        s.state_into(f=st["f"])
        return {"f": st["f"].float()}
    if c["kind"] == "adjoint":
        loss, ge, gs, gv = s.adjoint(c["steps"], c["ckpt"], dv0_out=st["out_v"])
        return {"scalars": np.array([loss, ge, gs], dtype=np.float32), "dv0": gv.float()}
    if c["kind"] == "dynamics":
        for _ in range(c["samples"]):
            s.integrate(c["steps"])
            s.dyn_sample()
        vacf, msd, _ = s.dyn_result()
        return {"vacf": vacf.astype(np.float32), "msd": msd.astype(np.float32), **_frame(st)}
    s.integrate(c["steps"])
    out = _frame(st)
    if c["props_every"]:
        rows = s.series(-(-c["steps"] // c["props_every"]))
        out["rows"] = rows if c["precision"] == "fp64" else rows.astype(np.float32)
    return out


def work(case):
    """Per step the state is read and written and the neighbour list read, per rebuild the list is
    written and the positions read; the frame is read and written once.  A pair of the list costs
    about 12 operations, one within r_c another 20."""
    c = case
    if c["kind"] == "batch":
        sizes = _replica_sizes(c)
        n = sum(k for k, _ in sizes)
        rho = sum(k * r for k, r in sizes) / n
    elif c["kind"] == "chains":
        n, rho = sum(e ** 3 for e in _replica_sizes(c)), c["rho"]
    elif c["kind"] == "dynamics":
        n, rho = c["nx"] * c["ny"] * c["nz"], c["rho"]
    else:
        n, rho = c["n"], c["rho"]
    reach = 4.0 / 3.0 * math.pi * rho
    listed_m, near_m = reach * (c["rc"] + c["skin"]) ** 3, reach * c["rc"] ** 3
    pair = 12.0 * listed_m + 20.0 * near_m
    if c["kind"] == "static":
        return {"bytes": n * (24.0 + 24.0 + 8.0), "flops": n * 32.0 * near_m}
    if c["kind"] == "forces":
        return {"bytes": n * (48.0 + 24.0 + 8.0 * listed_m), "flops": n * (pair + 10.0 * listed_m)}
    state = {"fp64": 48.0, "mixed": 48.0, "fp32": 24.0}[c["precision"]]
    steps = c["steps"] * c.get("samples", 1)
    every = 1.0 if c["rule"] == "every" else max(1.0, 0.5 * c["skin"] / (DT * 4.5 * math.sqrt(c["temp"])))
    rebuilds = steps / every
    b = n * (steps * (2.0 * state + 4.0 * listed_m) + rebuilds * (0.5 * state + 4.0 * listed_m) + 96.0)
    f = n * (steps * (pair + 12.0) + rebuilds * 10.0 * listed_m)
    if c["kind"] == "dynamics":
        b += n * c["samples"] * (72.0 + 48.0 * min(NLAG // ORIGIN_EVERY, 1 + c["samples"] // ORIGIN_EVERY))
    if c["kind"] == "adjoint":
        b, f = 3.0 * b, 4.0 * f        # forward, recompute and the reverse walk with its second derivatives
    return {"bytes": b, "flops": f}


# ---------------------------------------------------------------------------------------------
# the same in 64 bits, from plain torch operations
# ---------------------------------------------------------------------------------------------
_HALF = [o for o in itertools.product((-1, 0, 1), repeat=3) if o > (0, 0, 0)]
_CHUNK = 1 << 25


class _Ref:
    """Lennard-Jones pairs of all replicas by half-shell cell search, and leapfrog steps, in FP64."""

    def __init__(self, c, x, n_rep, boxes):
        self.c, self.boxes = c, boxes
        self.rep = torch.repeat_interleave(torch.arange(len(n_rep), device="cuda"),
                                           torch.tensor(n_rep, device="cuda"))
        self.n_rep, self.x_ref, self.i, self.j = n_rep, None, None, None

    def box_of(self, idx):
        return self.boxes[0] if len(self.n_rep) == 1 else self.boxes[self.rep[idx]]

    def gap(self, x, i, j):
        d = x[j] - x[i]
        b = self.box_of(i)
        return d - b * torch.round(d.detach() / b)

    def pairs(self, x):
        """Half list of the pairs within r_c + skin, kept until an atom may have moved skin / 2."""
        if self.x_ref is not None and self.c["skin"] > 0.0:
            d = x - self.x_ref
            b = self.box_of(slice(None))
            d = d - b * torch.round(d / b)
            if float((d * d).sum(1).max()) < (0.5 * self.c["skin"]) ** 2:
                return self.i, self.j
        reach = self.c["rc"] + self.c["skin"]
        nc = torch.floor(self.boxes / reach).long()
        ncell = nc.prod(1)
        base = torch.cumsum(ncell, 0) - ncell
        my_nc = nc[self.rep]
        cell = torch.minimum((x / self.boxes[self.rep] * my_nc).floor().long().clamp_(min=0), my_nc - 1)

        def number(q):
            return base[self.rep] + (q[:, 2] * my_nc[:, 1] + q[:, 1]) * my_nc[:, 0] + q[:, 0]

        cid = number(cell)
        order = torch.argsort(cid)
        count = torch.bincount(cid, minlength=int(ncell.sum()))
        start = torch.cumsum(count, 0) - count
        place = torch.empty_like(order)
        place[order] = torch.arange(order.numel(), device="cuda")
        found_i, found_j = [], []
        for off in [(0, 0, 0)] + _HALF:
            other = number(torch.remainder(cell + torch.tensor(off, device="cuda"), my_nc))
            first = place + 1 - start[other] if off == (0, 0, 0) else torch.zeros_like(place)
            left = count[other] - first
            for s in range(int(left.max())):
                i = torch.nonzero(left > s).squeeze(1)
                j = order[start[other[i]] + first[i] + s]
                d = self.gap(x, i, j)
                keep = (d * d).sum(1) < reach * reach
                found_i.append(i[keep].int())
                found_j.append(j[keep].int())
        self.i, self.j, self.x_ref = torch.cat(found_i), torch.cat(found_j), x.clone()
        return self.i, self.j

    def forces(self, x, per_atom_u=False):
        """(f, U per replica, virial per replica, u_i): u_i only where asked for."""
        c = self.c
        i_all, j_all = self.pairs(x)
        f = torch.zeros_like(x)
        u_atom = torch.zeros(x.shape[0] if per_atom_u else 0, dtype=torch.float64, device="cuda")
        U = torch.zeros(len(self.n_rep), dtype=torch.float64, device="cuda")
        W = torch.zeros_like(U)
        rc2 = c["rc"] ** 2
        uc = 4.0 * (rc2 ** -6 - rc2 ** -3)
        for k in range(0, i_all.numel(), _CHUNK):
            i, j = i_all[k:k + _CHUNK].long(), j_all[k:k + _CHUNK].long()
            d = self.gap(x, i, j)
            r2 = (d * d).sum(1)
            near = torch.nonzero(r2 < rc2).squeeze(1)
            i, j, d, r2 = i[near], j[near], d[near], r2[near]
            q6 = r2 ** -3
            g = 48.0 * q6 * (q6 - 0.5) / r2
            u = 4.0 * q6 * (q6 - 1.0) - uc
            f.index_add_(0, i, d * -g[:, None])
            f.index_add_(0, j, d * g[:, None])
            if len(self.n_rep) == 1:
                U += u.sum()
                W += (g * r2).sum()
            else:
                U.index_add_(0, self.rep[i], u)
                W.index_add_(0, self.rep[i], g * r2)
            if per_atom_u:
                u_atom.index_add_(0, i, u)
                u_atom.index_add_(0, j, u)
        if c["kind"] == "chains":
            f = f + self.chain_forces(x)
        return f, U, W, u_atom

    def chain_forces(self, x):
        x = x.detach().requires_grad_(True)
        local = torch.cat([torch.arange(n, device="cuda") for n in self.n_rep])
        size = torch.tensor(self.n_rep, device="cuda")[self.rep]
        idx = torch.arange(x.shape[0], device="cuda")
        m = CHAIN["length"]
        a = idx[(local % m < m - 1) & (local < size - 1)]
        b2 = (self.gap(x, a, a + 1) ** 2).sum(1)
        r02 = CHAIN["fene_r0"] ** 2
        e = (-0.5 * CHAIN["fene_k"] * r02 * torch.log(1.0 - b2 / r02)).sum()
        a = idx[(local % m < m - 2) & (local < size - 2)]
        b, d = self.gap(x, a, a + 1), self.gap(x, a + 1, a + 2)
        e = e + (CHAIN["bend_k"] * (1.0 - (b * d).sum(1) / torch.sqrt((b * b).sum(1) * (d * d).sum(1)))).sum()
        return -torch.autograd.grad(e, x)[0]

    def kinetic(self, v):
        k = 0.5 * (v * v).sum(1)
        out = torch.zeros(len(self.n_rep), dtype=torch.float64, device="cuda")
        return out + k.sum() if len(self.n_rep) == 1 else out.index_add_(0, self.rep, k)

    def step(self, x, v, f):
        v = v + 0.5 * DT * f
        x = _wrapped(x + DT * v, self.box_of(slice(None)))
        f, U, W, _ = self.forces(x)
        return x, v + 0.5 * DT * f, f, U, W


def _exact_adjoint(c, x0, v0, box, n_rep):
    ref = _Ref(c, x0, n_rep, box)
    b = box[0]
    eps = torch.tensor(1.0, dtype=torch.float64, device="cuda", requires_grad=True)
    sig = torch.tensor(1.0, dtype=torch.float64, device="cuda", requires_grad=True)
    v0 = v0.clone().requires_grad_(True)

    def pair(x):
        i, j = (t.long() for t in ref.pairs(_wrapped(x.detach(), b)))
        d = ref.gap(x, i, j)
        r2 = (d * d).sum(1)
        near = torch.nonzero(r2.detach() < c["rc"] ** 2).squeeze(1)
        i, j, d, r2 = i[near], j[near], d[near], r2[near]
        q6 = (sig * sig / r2) ** 3
        g = 48.0 * eps * q6 * (q6 - 0.5) / r2
        f = torch.zeros_like(x).index_add(0, i, d * -g[:, None]).index_add(0, j, d * g[:, None])
        return f, (4.0 * eps * q6 * (q6 - 1.0) + eps).sum()

    x, v, total = x0, v0, 0.0
    f, _ = pair(x)
    for _ in range(c["steps"]):
        v = v + 0.5 * DT * f
        x = x + DT * v
        f, u = pair(x)
        v = v + 0.5 * DT * f
        total = total + u
    loss = total / c["steps"] + (v * v).sum()
    ge, gs, gv = torch.autograd.grad(loss, (eps, sig, v0))
    return {"scalars": np.array([float(loss), float(ge), float(gs)]), "dv0": gv}


def exact(case, seed):
    c = dict(case)
    w = work(c)
    if w["flops"] > 2.0e11:            # the largest systems: the pair arithmetic below takes too long
        return None
    x, v, n_rep, boxes = _state(c, seed)
    if c["kind"] == "static":
        c["skin"] = 0.0
    if c["kind"] == "forces":
        x, v, n_rep, boxes = _state(c, int(seed) + 500009)
    if c["kind"] == "adjoint":
        return _exact_adjoint(c, x, v, boxes, n_rep)
    ref = _Ref(c, x, n_rep, boxes)
    f, U, W, u = ref.forces(x, per_atom_u=c["kind"] == "static")
    if c["kind"] == "static":
        return {"f": f, "u": u}
    if c["kind"] == "forces":
        return {"f": f}
    if c["kind"] == "dynamics":
        vacf, msd = np.zeros(NLAG), np.zeros(NLAG)
        moved, v0 = torch.zeros_like(x), None
        for s in range(c["samples"]):
            for _ in range(c["steps"]):
                y = x
                x, v, f, _, _ = ref.step(x, v, f)
                d = x - y
                moved += d - boxes[0] * torch.round(d / boxes[0])
            if s == 0:                                   # the one time origin of the first samples
                v0, moved = v.clone(), torch.zeros_like(x)
            vacf[s] = float((v * v0).sum()) / n_rep[0]
            msd[s] = float((moved * moved).sum()) / n_rep[0]
        return {"vacf": vacf, "msd": msd, "x": x, "v": v}
    rows = []
    volume = boxes.prod(1)
    for k in range(c["steps"]):
        if c["props_every"] and k % c["props_every"] == 0:
            K = ref.kinetic(v)
            P = torch.stack([v[ref.rep == r].sum(0) for r in range(len(n_rep))])
            vmax = torch.stack([(v[ref.rep == r] ** 2).sum(1).max().sqrt() for r in range(len(n_rep))])
            rows.append(torch.cat([torch.full_like(K, float(k))[:, None], U[:, None], K[:, None], W[:, None],
                                   ((2.0 * K + W) / (3.0 * volume))[:, None], P, vmax[:, None]], 1))
        x, v, f, U, W = ref.step(x, v, f)
    out = {"x": x, "v": v}
    if rows:
        out["rows"] = torch.stack(rows, 1)
    return out
