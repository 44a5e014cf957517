"""Paths that only some sizes, shapes or options take: warp-tiles claimed and stolen (named shapes of few
warps; FP64 beyond 40 warp-tiles per SM), the gathered reorder (above 2048 tiles), the scan in three
kernels with the chunks of replicas at rest passed over (above 65536 cells), and the state read through
the half list or with chain terms."""
import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
from paper_2003_14061_gb300 import binding as B
from paper_2003_14061_gb300 import inputs
from paper_2003_14061_gb300.system import WCA_RC, MDSystem

pytestmark = pytest.mark.gpu
PRECS = ["fp64", "mixed", "fp32"]


def min_image(d, box):
    return d - box * np.round(d / box)


@pytest.mark.parametrize("prec", PRECS)
@pytest.mark.parametrize("rule", ["vmax", "disp"])
def test_claimed_warp_tiles_give_the_same_bits(prec, rule):
    # 1000 warp-tiles: a warp each by default; 152 CTAs of 4 warps claim them
    x, box = inputs.fcc_lattice(20, 0.8)
    x = inputs.perturb(x, box, 0.1, 1)
    v = inputs.maxwell(x.shape[0], 1.0, 2)
    out = []
    for tuning in ({}, dict(ctas_per_sm=1), dict(ctas_per_sm=1, nbr_batch=8)):
        s = MDSystem(x, v, box, skin=0.4, precision=prec, rebuild_rule=rule, props_every=1)
        if tuning:
            s.set_tuning(**tuning)
        s.integrate(48)
        out.append((*s.state(f=True), s.series(64)))
        assert s.props()[0]["rebuilds"] > 2
    for other in out[1:]:
        for a, b in zip(out[0], other):
            assert np.array_equal(a, b)


@pytest.mark.parametrize("prec", PRECS)
def test_gathered_reorders_match_oracle(prec):
    x, box = inputs.fcc_lattice(41, 0.8)               # 275684 atoms, 2154 tiles
    x = inputs.perturb(x, box, 0.1, 3)
    n = x.shape[0]
    v = inputs.maxwell(n, 1.0, 4)
    s = MDSystem(x, v, box, skin=0.4, precision=prec, reorder_every=0, props_every=1)
    s.integrate(20)
    xg, vg, fg = s.state(f=True)
    pr = s.props()[0]
    xo, vo, po, _ = oracle.run(x, v, box, oracle.pot(rc=WCA_RC), dt=0.005, nsteps=20, rule=1, skin=0.4)
    assert pr["reorders"] == pr["rebuilds"] >= 2
    assert np.abs(min_image(xg - xo, box)).max() <= (1e-9 if prec == "fp64" else 1e-4)
    assert np.abs(vg - vo).max() <= (1e-8 if prec == "fp64" else 1e-2)
    ser = s.series(32)[0]
    assert np.abs((ser[:, 1] + ser[:, 2]) - (po[:20, 0] + po[:20, 1])).max() / n <= 1e-6


@pytest.mark.parametrize("prec", PRECS)
def test_batch_scan_passes_over_replicas_at_rest(prec):
    # 100 replicas of 729 cells each, hotter and hotter, so that they rebuild at steps of their own;
    # batches of 20 of them are scanned in one kernel
    nrep, parts = 100, 5
    xs, vs, boxes = [], [], []
    for r in range(nrep):
        x, box = inputs.fcc_lattice(8 if r % 3 else 7, 0.8)
        xs.append(inputs.perturb(x, box, 0.1, r))
        vs.append(inputs.maxwell(x.shape[0], 0.3 + 0.03 * r, r))
        boxes.append(np.array([13.69, 13.69, 13.69]) if r % 3 else box)

    def run(a, b):
        s = MDSystem(np.concatenate(xs[a:b]), np.concatenate(vs[a:b]), n_rep=[len(x) for x in xs[a:b]],
                     boxes=np.array(boxes[a:b]), skin=0.4, precision=prec, cell_block=1, reorder_every=20, nbr_capacity=40)
        s.integrate(40)
        return s.state()[:2], [(p["rebuilds"], p["reorders"], p["max_nbrs"], p["max_cell_occ"]) for p in s.props()]

    (x, v), counts = run(0, nrep)
    assert len({c[0] for c in counts}) > 4
    step = nrep // parts
    small = [run(k * step, (k + 1) * step) for k in range(parts)]
    assert np.array_equal(x, np.concatenate([q[0][0] for q in small]))
    assert np.array_equal(v, np.concatenate([q[0][1] for q in small]))
    assert counts == [c for q in small for c in q[1]]


@pytest.mark.parametrize("prec", ["mixed", "fp32"])
@pytest.mark.parametrize("kernel,chains", [(5, False), (1, True), (4, True), (5, True)])
@pytest.mark.parametrize("ncell", [5, 30])
def test_state_of_half_list_and_chains_in_every_memory(prec, kernel, chains, ncell):
    x, box = inputs.fcc_lattice(ncell, 0.8)
    x = inputs.perturb(x, box, 0.05, 1)
    n = x.shape[0]
    s = MDSystem(x, inputs.maxwell(n, 0.5, 2), box, skin=0.3, precision=prec)
    if kernel != 1:
        s.set_tuning(step_kernel=kernel)
    if chains:
        s.set_chains(1, 30.0, 1.5)                     # chains of single atoms: the buffers are used, their terms are zero
    s.integrate(7)
    want = s.state(f=True)                             # host arrays, through the exchange buffers
    ref = MDSystem(want[0], want[1], box, skin=0.3, precision=prec).state(x=False, v=False, f=True)[2]
    buf = torch.full((3 * 3 * n + 1,), float("nan"), dtype=torch.float64, device="cuda")
    parts = [buf[1 + 3 * n * q: 1 + 3 * n * (q + 1)].view(n, 3) for q in range(3)]     # 8-byte aligned only

    def get(*t):
        B.call("md_get_state", s.h, *[None if a is None else ctypes.c_void_p(a.data_ptr()) for a in t])

    def same(q, got):
        got = got.cpu().numpy()
        if q == 0 or kernel != 5:
            assert np.array_equal(got, want[q])
        else:                                          # the half list adds in no fixed order
            assert np.linalg.norm(got - want[q]) <= 1e-5 * np.linalg.norm(want[q])

    get(*parts)
    for q in range(3):
        same(q, parts[q])
    for q in range(3):                                 # one array at a time, and the buffers are left at zero
        out = torch.full((n, 3), float("nan"), dtype=torch.float64, device="cuda")
        get(*[out if k == q else None for k in range(3)])
        same(q, out)
    pin = torch.empty(n, 3, dtype=torch.float64, pin_memory=True)
    get(None, pin, parts[2])
    same(1, pin)
    same(2, parts[2])
    assert np.linalg.norm(want[2] - ref) <= 1e-3 * np.linalg.norm(ref)
