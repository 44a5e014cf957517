"""Neighbour columns that the build's lists do not hold: a warp then writes the atom's column itself.

Dense clusters in boxes of a low mean density (lists are sized for the mean and, up to 84 rows, for the
capacity) and runs of more candidates than a list entry can number; the oracle's sets, in the order
rows of cells, cells, slots, at box boundaries too, for the full and the half list."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
from paper_2003_14061_gb300.system import MDSystem

pytestmark = pytest.mark.gpu
RC, SKIN = 1.1, 0.4


def _cluster(n, centre, box, spread, seed):
    return np.mod(np.array(centre) + np.random.default_rng(seed).uniform(-spread, spread, (n, 3)), box)


def _case(name):
    """(positions, box, capacity)"""
    rng = np.random.default_rng(8)
    if name == "clusters":               # in the middle of a cell, on faces, on a corner of the box
        box = np.array([18.3, 21.4, 24.0])
        parts = [rng.uniform(0, 1, (200, 3)) * box]
        for k, c in enumerate([(9.0, 9.0, 9.0), (0.0, 7.0, 15.0), (18.3, 0.0, 20.0), (0.0, 0.0, 0.0)]):
            parts.append(_cluster(150 + 31 * k, c, box, 0.6, k))
        return np.concatenate(parts), box, 420
    if name == "three_cells":            # every row of cells reached across the boundary; all units overflow
        box = np.array([4.7, 4.8, 4.6])
        return rng.uniform(0, 1, (900, 3)) * box, box, 400
    if name == "long_run":               # 4216 candidates in the run of the middle cell's atoms, none near them
        box = np.array([7.7, 4.8, 4.8])  # 5 x 3 x 3 cells of 1.54 x 1.6 x 1.6
        a = np.array([1.56, 2.4, 2.4]) + rng.uniform(0, 1, (2100, 3)) * (0.01, 0.5, 0.5)
        b = np.array([6.13, 2.4, 2.4]) + rng.uniform(0, 1, (2104, 3)) * (0.01, 0.5, 0.5)
        mid = np.array([3.1, 2.4, 2.4]) + rng.uniform(0, 1, (12, 3)) * (1.5, 0.5, 0.5)
        return np.concatenate([a, mid, b]), box, 2110
    raise KeyError(name)


def _place(cell, nc):
    """for each atom, its cell's coordinates"""
    return np.stack([cell % nc[0], cell // nc[0] % nc[1], cell // (nc[0] * nc[1])], -1)


@pytest.mark.parametrize("prec", ["fp64", "mixed", "fp32"])
@pytest.mark.parametrize("name", ["clusters", "three_cells", "long_run"])
def test_long_columns(name, prec):
    x, box, cap = _case(name)
    n = len(x)
    s = MDSystem(x, np.zeros_like(x), box, rc=RC, skin=SKIN, precision=prec, nbr_capacity=cap, cell_block=1)
    nc, cell = oracle.cells(x, box, RC + SKIN)
    c = _place(np.asarray(cell), np.asarray(nc))
    _, oc, off, onb = oracle.neighbours(x, box, RC, SKIN, fp32=(prec != "fp64"))
    assert oc.max() <= cap and oc.max() > 150
    counts, nb = s.neighbours()
    assert np.array_equal(counts, oc)
    for i in range(n):
        got = nb[i, : counts[i]]
        assert np.array_equal(np.sort(got), onb[off[i]: off[i + 1]]), i
        o = (c[got] - c[i] + 1) % np.asarray(nc)                       # 0, 1, 2 along each axis
        key = ((o[:, 2] * 3 + o[:, 1]) * 3 + o[:, 0]) * np.int64(n) + got
        assert np.all(np.diff(key) > 0), i
    if prec == "fp64":
        return
    s.set_tuning(step_kernel=5)                                        # each pair once
    half, nb = s.neighbours()
    seen = [set() for _ in range(n)]
    for i in range(n):
        for j in nb[i, : half[i]]:
            seen[i].add(int(j))
            seen[int(j)].add(i)
    assert 2 * int(half.sum()) == int(oc.sum())
    assert all(len(q) == k for q, k in zip(seen, oc))
    assert all(q == set(onb[off[i]: off[i + 1]].tolist()) for i, q in enumerate(seen))
