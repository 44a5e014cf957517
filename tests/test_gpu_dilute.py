"""Boxes with far more cells than atoms: the cells' bookkeeping leaves the tiles of atoms.

A tile of 128 slots does up to 256 cells of its replica itself; beyond, all CTAs share the cells in
chunks of 512.  Sizes either side of both, and batches in which only some replicas are so."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
from paper_2003_14061_gb300 import inputs
from paper_2003_14061_gb300.system import WCA_RC, MDSystem

pytestmark = pytest.mark.gpu
RC, SKIN = 1.1, 0.4


def _atoms(n, cells, seed):
    """n atoms in pairs and triples (so that there are neighbours) in a box of the given cells."""
    rng = np.random.default_rng(seed)
    box = (np.array(cells) + 0.5) * (RC + SKIN)
    x = rng.uniform(0.0, 1.0, (n, 3)) * box
    for i in range(1, n):
        if i % 3:
            x[i] = np.mod(x[i - 1] + rng.uniform(0.3, 0.8, 3), box)
    return x, box


def _same_sets(x, box, counts, nb, base, prec):
    _, oc, off, onb = oracle.neighbours(x, box, RC, SKIN, fp32=(prec != "fp64"))
    assert np.array_equal(counts, oc)
    for i in range(len(x)):
        assert np.array_equal(np.sort(nb[i, : oc[i]]) - base, onb[off[i]: off[i + 1]]), i


@pytest.mark.parametrize("prec", ["fp64", "mixed", "fp32"])
@pytest.mark.parametrize("n,cells", [(1, (7, 7, 6)), (100, (4, 8, 8)), (100, (257, 3, 3)), (129, (3, 9, 19)),
                                     (128, (16, 8, 4)), (7, (50, 41, 30)), (300, (70, 70, 40))])
def test_sets_of_dilute_systems(prec, n, cells):
    x, box = _atoms(n, cells, n)
    s = MDSystem(x, np.zeros_like(x), box, rc=RC, skin=SKIN, precision=prec, nbr_capacity=24)
    assert tuple(s.cells_per_axis()) == cells
    for _ in range(2):                            # the second one finds the counters cleared
        counts, nb = s.neighbours()
        _same_sets(x, box, counts, nb, 0, prec)
        s.build_neighbours()
    assert s.props()[0]["max_cell_occ"] == np.bincount(oracle.cells(x, box, RC + SKIN)[1]).max()


@pytest.mark.parametrize("kernel", [1, 4])
def test_batch_with_dilute_and_dense_replicas(kernel):
    # every replica rebuilds at steps of its own; the dense ones give the trajectory of the oracle, the
    # dilute ones, whose atoms never meet, move on straight lines
    xs, vs, boxes = [], [], []
    for r, kind in enumerate("dgdggd"):
        if kind == "d":
            x, box = inputs.fcc_lattice(4 + r % 3, 0.8)
            x, v = inputs.perturb(x, box, 0.1, r), inputs.maxwell(x.shape[0], 1.0, 20 + r)
        else:
            m = 6 + r
            box = np.array([40.0, 50.0 + r, 60.0])
            g = np.stack(np.meshgrid(*[np.arange(m)] * 3, indexing="ij"), -1).reshape(-1, 3)[: 5 * m * m + 1]
            x = (g + 0.5) * box / m
            v = np.random.default_rng(r).normal(0.0, 1.0 + r, x.shape).clip(-4, 4)
        xs.append(x)
        vs.append(v)
        boxes.append(box)
    s = MDSystem(np.concatenate(xs), np.concatenate(vs), n_rep=[len(x) for x in xs], boxes=np.array(boxes), rc=WCA_RC,
                 skin=0.4, precision="mixed", nbr_capacity=40)
    if kernel != 1:
        s.set_tuning(step_kernel=kernel)
    s.integrate(60)
    xg, _, _ = s.state()
    pr = s.props()
    assert len({p["rebuilds"] for p in pr}) > 2
    off = 0
    for x, v, box in zip(xs, vs, boxes):
        if np.prod(box) > 1e5:
            want = np.mod(x + 60 * 0.005 * v, box)
        else:
            want, _, _, _ = oracle.run(x, v, box, oracle.pot(rc=WCA_RC), dt=0.005, nsteps=60, with_props=False)
        d = xg[off: off + len(x)] - want
        assert np.abs(d - box * np.round(d / box)).max() <= 1e-4
        off += len(x)
