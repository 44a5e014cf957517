"""State exchange through device, host and mixed arrays: the same bits whichever memory the caller's
arrays are in, aligned or not to anything but doubles, one array or several, and with arrays that
share memory (copied one after the other, as documented order x, v, f)."""
import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2003_14061_gb300 import binding as B
from paper_2003_14061_gb300 import inputs
from paper_2003_14061_gb300.system import MDSystem

pytestmark = pytest.mark.gpu


def _get(s, x=None, v=None, f=None):
    B.call("md_get_state", s.h, *[None if t is None else ctypes.c_void_p(t.data_ptr()) for t in (x, v, f)])


@pytest.mark.parametrize("kernel", [1, 4, 5])
@pytest.mark.parametrize("prec", ["fp64", "mixed", "fp32"])
@pytest.mark.parametrize("ncell", [4, 14])
def test_same_bits_from_every_memory(prec, kernel, ncell):
    x, box = inputs.fcc_lattice(ncell, 0.8)
    x = inputs.perturb(x, box, 0.1, seed=1)
    v = inputs.maxwell(x.shape[0], 1.0, seed=2)
    n = x.shape[0]
    a = MDSystem(x, v, box, precision=prec, skin=0.4)
    b = MDSystem(torch.from_numpy(x).cuda(), torch.from_numpy(v).cuda(), box, precision=prec, skin=0.4)
    for s in (a, b):
        if prec != "fp64" and kernel != 5:               # the half list adds in no fixed order
            s.set_tuning(step_kernel=kernel)
        s.integrate(17)
    xa, va, fa = a.state(f=True)
    buf = torch.full((3 * 3 * n + 1,), float("nan"), dtype=torch.float64, device="cuda")
    parts = [buf[1 + 3 * n * q: 1 + 3 * n * (q + 1)].view(n, 3) for q in range(3)]     # 8-byte aligned only
    _get(b, *parts)
    for got, want in zip(parts, (xa, va, fa)):
        assert np.array_equal(got.cpu().numpy(), want)
    for q, want in enumerate((xa, va, fa)):              # one array at a time
        out = torch.full((n, 3), float("nan"), dtype=torch.float64, device="cuda")
        _get(b, *[out if k == q else None for k in range(3)])
        assert np.array_equal(out.cpu().numpy(), want)
    pin = torch.empty(n, 3, dtype=torch.float64, pin_memory=True)
    dev = torch.empty(n, 3, dtype=torch.float64, device="cuda")
    _get(b, pin, dev, None)                              # host and device together
    assert np.array_equal(pin.numpy(), xa) and np.array_equal(dev.cpu().numpy(), va)
    both = torch.empty(n, 3, dtype=torch.float64, device="cuda")
    _get(b, both, both, None)                            # the same array twice: the later copy stays
    assert np.array_equal(both.cpu().numpy(), va)
    a.set_state(xa, va)
    b.set_state(torch.from_numpy(xa).cuda(), torch.from_numpy(va).cuda())
    for s in (a, b):
        s.integrate(5)
    assert np.array_equal(a.state()[0], b.state()[0])
