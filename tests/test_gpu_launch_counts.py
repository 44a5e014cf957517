"""Kernels that md_get_timing counts for the calls outside a step, against what each call launches:
pairs (half list: and their sums into the force array), chain terms before them, the kernels that use
the forces."""
import pytest

torch = pytest.importorskip("torch")

from paper_2003_14061_gb300 import inputs
from paper_2003_14061_gb300.system import MDSystem

pytestmark = pytest.mark.gpu


def _count(s, phase, f):
    s.timing()                                     # resets the counters
    f()
    return s.timing()[phase][2]


@pytest.mark.parametrize("prec,kernel,chains,forces", [("fp64", 1, False, 1), ("mixed", 1, False, 1), ("fp32", 4, False, 1),
                                                       ("mixed", 5, False, 2), ("mixed", 1, True, 2), ("fp32", 4, True, 2),
                                                       ("fp32", 5, True, 3)])
def test_counted_launches(prec, kernel, chains, forces):
    x, box = inputs.fcc_lattice(5, 0.5)
    s = MDSystem(x, inputs.maxwell(x.shape[0], 1.0, 2), box, skin=0.3, precision=prec)
    if kernel != 1:
        s.set_tuning(step_kernel=kernel)
    if chains:
        s.set_chains(1, 30.0, 1.5)
    # in one pass where the forces come from one kernel, else the forces and a kernel that reads them
    get = 1 if forces == 1 else forces + 1
    assert _count(s, "other", lambda: s.state(v=False)) == 1
    assert _count(s, "other", lambda: s.state(f=True)) == get
    assert _count(s, "other", s.compute_forces) == forces
    assert _count(s, "props", s.props) == forces + 2
    s.dyn_begin(4, 2)
    assert _count(s, "other", s.dyn_sample) == forces + 2
