"""An atom whose position is no longer finite stays its own replica's matter.

Replica 0 of a batch is two atoms, at one point (their force is 0 / 0) or apart; the other replicas
are the same fluids in both runs.  Every state, force and measured quantity of those must be the
same bits: columns of W are padded to whole batches of entries, and what pads them must not bring
another replica's position in."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2003_14061_gb300 import binding as B
from paper_2003_14061_gb300 import inputs
from paper_2003_14061_gb300.system import WCA_RC, MDSystem

pytestmark = pytest.mark.gpu

SHAPES = [dict(), dict(ctas_per_sm=4, nbr_batch=8), dict(ctas_per_sm=8, nbr_batch=4), dict(ctas_per_sm=8, nbr_batch=2),
          dict(step_kernel=2, nbr_batch=8), dict(step_kernel=3, nbr_batch=8), dict(step_kernel=4), dict(step_kernel=5)]


def _run(prec, tuning, apart):
    pair = np.array([[2.0, 2.0, 2.0], [2.0 + apart, 2.0, 2.0]])
    xs, boxes = [pair], [np.array([6.0, 6.0, 6.0])]
    for k, n in enumerate((5, 6)):
        x, box = inputs.fcc_lattice(n, 0.8)
        xs.append(inputs.perturb(x, box, 0.1, 30 + k))
        boxes.append(box)
    sizes = [len(x) for x in xs]
    v = np.concatenate([np.zeros((2, 3))] + [inputs.maxwell(n, 1.0, 40 + n) for n in sizes[1:]])
    s = MDSystem(np.concatenate(xs), v, n_rep=sizes, boxes=np.array(boxes), rc=WCA_RC, skin=0.4, precision=prec,
                 props_every=1, nbr_capacity=64)
    if tuning:
        s.set_tuning(**tuning)
    s.integrate(37)
    bad = False
    try:
        s.check()
    except B.MDError as e:
        bad = "non-finite" in str(e)
    assert bad == (apart == 0.0)
    out = s.state(f=True)
    rows = s.series(64)
    return [a[2:] for a in out] + [rows[1:]]


@pytest.mark.parametrize("prec,tuning", [(p, t) for p in ("fp64", "mixed", "fp32") for t in SHAPES
                                         if p != "fp64" or not t])
def test_other_replicas_are_untouched(prec, tuning):
    good, got = _run(prec, tuning, 1.5), _run(prec, tuning, 0.0)
    for a, b in zip(good, got):
        assert np.isfinite(b).all()
        if tuning.get("step_kernel") == 5:        # the half list adds in no fixed order
            assert np.allclose(a, b, rtol=0, atol=1e-2 * max(1.0, np.abs(a).max()))
        else:
            assert np.array_equal(a, b)
