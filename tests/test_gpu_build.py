"""GPU tests of the neighbour build at the sizes where its units, rows and lists end.

The build scans the three z planes around an atom into three lists and joins them, so the inputs
are boxes of three cells along some axis (every row of cells is reached across the boundary too),
rows of cells with no atoms, replicas of a few atoms and of one more than a unit or a tile, and a
cluster whose lists overflow.  The sets are the oracle's, bit for bit; the order of a column is
rows of cells, cells, then slots, written out here in plain Python."""
import numpy as np
import pytest

import oracle
from paper_2003_14061_gb300 import inputs
from paper_2003_14061_gb300.system import MDSystem

pytestmark = pytest.mark.gpu
PRECS = ["fp64", "mixed", "fp32"]


def _uniform(n, box, seed):
    return np.random.default_rng(seed).uniform(0.0, 1.0, (n, 3)) * np.asarray(box)


def _case(name):
    """(positions, box, r_c, skin, capacity)"""
    if name == "three_cells":                # every neighbouring cell is its own periodic image's neighbour
        return _uniform(211, (4.6, 4.6, 4.6), 1), (4.6, 4.6, 4.6), 1.1, 0.4, 120
    if name == "flat":                       # 3 x 17 x 4 cells
        return _uniform(700, (4.7, 25.7, 6.3), 2), (4.7, 25.7, 6.3), 1.1, 0.4, 60
    if name == "gas":                        # most cells and many rows of cells are empty
        return _uniform(131, (31.0, 19.0, 23.0), 3), (31.0, 19.0, 23.0), 1.1, 0.4, 20
    if name == "cluster":                    # 260 atoms within r_c + skin of each other: lists overflow
        x = _uniform(300, (12.0, 12.0, 12.0), 4)
        x[:260] = 5.0 + _uniform(260, (0.8, 0.8, 0.8), 5)
        return x, (12.0, 12.0, 12.0), 1.1, 0.4, 300
    n = int(name)                            # a unit, a tile, and one atom either side
    x, box = inputs.fcc_subset(n, 0.8, seed=n) if n > 200 else (_uniform(n, (6.1, 6.1, 6.1), n), (6.1, 6.1, 6.1))
    return x, tuple(box), 1.1, 0.4, 0


def _expected_order(x, box, rl, i, members, cell, nc):
    """members of atom i's column in the order rows of cells (z, then y), cells, ids."""
    c = np.array([cell[i] % nc[0], (cell[i] // nc[0]) % nc[1], cell[i] // (nc[0] * nc[1])])
    place = {}
    k = 0
    for oz in (-1, 0, 1):
        for oy in (-1, 0, 1):
            for ox in (-1, 0, 1):
                q = (c + np.array([ox, oy, oz])) % nc
                place[int((q[2] * nc[1] + q[1]) * nc[0] + q[0])] = k
                k += 1
    return sorted(members, key=lambda j: (place[int(cell[j])], j))


@pytest.mark.parametrize("prec", PRECS)
@pytest.mark.parametrize("name", ["three_cells", "flat", "gas", "cluster", "9", "10", "11", "127", "128", "129", "1031"])
def test_columns(name, prec):
    x, box, rc, skin, cap = _case(name)
    v = np.zeros_like(x)
    s = MDSystem(x, v, np.array(box), rc=rc, skin=skin, precision=prec, nbr_capacity=cap, cell_block=1)
    counts, nb = s.neighbours()
    nc, cell = oracle.cells(x, np.array(box), rc + skin)
    _, oc, off, onb = oracle.neighbours(x, np.array(box), rc, skin, fp32=(prec != "fp64"))
    assert np.array_equal(counts, oc)
    nc = np.asarray(nc)
    for i in range(x.shape[0]):
        want = onb[off[i]: off[i + 1]]
        assert list(nb[i, : counts[i]]) == _expected_order(x, box, rc + skin, i, list(want), cell, nc), i
    pr = s.props()[0]
    assert pr["max_nbrs"] == oc.max() and abs(pr["mean_nbrs"] - oc.mean()) <= 1e-9
    assert pr["max_cell_occ"] == np.bincount(cell).max()


@pytest.mark.parametrize("prec", PRECS)
def test_replicas_of_a_few_atoms(prec):
    sizes = [1, 2, 10, 127, 129, 31]
    xs = [_uniform(n, (5.1, 6.2, 7.9), 50 + n) for n in sizes]
    s = MDSystem(np.concatenate(xs), np.zeros((sum(sizes), 3)), n_rep=sizes,
                 boxes=np.tile([5.1, 6.2, 7.9], (len(sizes), 1)), rc=1.1, skin=0.4, precision=prec, nbr_capacity=64)
    counts, nb = s.neighbours()
    base = 0
    for x in xs:
        _, oc, off, onb = oracle.neighbours(x, np.array([5.1, 6.2, 7.9]), 1.1, 0.4, fp32=(prec != "fp64"))
        assert np.array_equal(counts[base: base + len(x)], oc)
        for i in range(len(x)):
            assert np.array_equal(np.sort(nb[base + i, : oc[i]]) - base, onb[off[i]: off[i + 1]])
        base += len(x)
