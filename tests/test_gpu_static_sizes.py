"""md_forces_static at the sizes where its paths end: one atom, boxes of three cells along an axis,
the largest system of the one-kernel cell list and the smallest of the separate kernels, and many
empty cells.  Forces and u_i against the FP64 oracle at the FP32 bars (1e-5), repeated calls bit for
bit; a call with another cell count in between leaves nothing behind."""
import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
from paper_2003_14061_gb300 import binding as B
from paper_2003_14061_gb300 import inputs
from paper_2003_14061_gb300.system import make_params

pytestmark = pytest.mark.gpu


def _call(x, box, rc):
    n = x.shape[0]
    p = make_params(n=n, box=box, rc=rc)
    xd = torch.from_numpy(np.ascontiguousarray(x)).to("cuda")
    fd = torch.full_like(xd, float("nan"))
    ud = torch.full((n,), float("nan"), dtype=torch.float64, device="cuda")
    B.call("md_forces_static", ctypes.byref(p), n, ctypes.c_void_p(xd.data_ptr()), ctypes.c_void_p(fd.data_ptr()),
           ctypes.c_void_p(ud.data_ptr()), ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    torch.cuda.synchronize()
    return fd.cpu().numpy(), ud.cpu().numpy()


@pytest.mark.parametrize("n,cells,rc", [(1, (5, 5, 5), 1.12), (32, (2, 2, 2), 1.1), (33, (3, 3, 3), 1.1), (500, (5, 5, 5), 2.5),
                                        (1997, (4, 9, 14), 1.12), (8192, (16, 8, 16), 1.12),
                                        (8193, (13, 13, 13), 1.12), (30000, (21, 19, 19), 2.5)])
def test_sizes(n, cells, rc):
    nx, ny, nz = cells
    x, _ = inputs.fcc_lattice(max(cells), 0.7)          # spacing only: the box is cut to nx x ny x nz cells
    a = (4.0 / 0.7) ** (1.0 / 3.0)
    keep = np.all(x < np.array(cells) * a, axis=1)
    box = np.array(cells) * a
    x = inputs.perturb(x[keep][:n], box, 0.1, seed=n)
    assert x.shape[0] == n
    f, u = _call(x, box, rc)
    of, ou, _, _ = oracle.forces(x, box, oracle.pot(rc=rc))
    scale = np.linalg.norm(of)
    assert np.linalg.norm(f - of) <= 1e-5 * (scale if scale > 0 else 1.0)
    assert np.abs(u - ou).max() <= 1e-5 * (np.abs(ou).max() + 1.0)
    _call(x[: max(1, n // 3)], box * 1.3, rc)
    f2, u2 = _call(x, box, rc)
    assert np.array_equal(f, f2) and np.array_equal(u, u2)
