"""The step kernel's launch shape: tuning that is read and written back, or named and put back to the
values of a new system, leaves the shape that the library chooses by size.

The shapes are those that the profiler records (kernel, grid, block), in a child process so that the
profiler stays out of this one."""
import json
import os
import subprocess
import sys

import pytest

pytest.importorskip("torch")
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
pytestmark = pytest.mark.gpu

CHILD = """
import json
import sys
import tempfile
import torch
from torch.profiler import profile, ProfilerActivity
from paper_2003_14061_gb300 import inputs
from paper_2003_14061_gb300.system import MDSystem

ncell, lj, prec = int(sys.argv[1]), sys.argv[2] == "lj", sys.argv[3]

def system():
    x, box = inputs.fcc_lattice(ncell, 0.8442 if lj else 0.8)
    v = inputs.maxwell(x.shape[0], 1.0, 2)
    return MDSystem(x, v, box, precision=prec, **(dict(rc=2.5, skin=0.3) if lj else dict(skin=0.4)))

def shape(s):
    s.set_tuning(use_graph=2)
    for _ in range(4):                        # the first session of a process may record nothing
        with profile(activities=[ProfilerActivity.CUDA]) as prof:
            s.integrate(1)
            torch.cuda.synchronize()
        with tempfile.NamedTemporaryFile(suffix=".json") as f:
            prof.export_chrome_trace(f.name)
            ev = json.load(open(f.name))["traceEvents"]
        got = [(e["name"].split("(")[0], e["args"]["grid"], e["args"]["block"]) for e in ev
               if "k_step" in e.get("name", "") and "grid" in e.get("args", {})]
        if got:
            return got
    raise RuntimeError("the profiler recorded no kernels")

a = system()
out = {"new": shape(a)}
a.set_tuning(**a.tuning())
out["written back"] = shape(a)
t = {k: a.tuning()[k] for k in ("ctas_per_sm", "nbr_batch")}
a.set_tuning(ctas_per_sm=12, nbr_batch=4)
out["named"] = shape(a)
a.set_tuning(**t)
out["put back"] = shape(a)
b = system()
b.set_tuning(**{k: system().tuning()[k] for k in ("ctas_per_sm", "nbr_batch", "build_batch", "build_stage",
                                                  "step_kernel", "reorder_every")})
out["copied"] = shape(b)
print(json.dumps(out))
"""


@pytest.mark.parametrize("ncell,fluid,prec", [(8, "wca", "mixed"), (10, "lj", "fp32"), (30, "wca", "mixed"), (30, "wca", "fp64"),
                                              (40, "lj", "mixed")])
def test_shape_by_size_survives_reading_and_writing(ncell, fluid, prec):
    r = subprocess.run([sys.executable, "-c", CHILD, str(ncell), fluid, prec], cwd=ROOT, capture_output=True, text=True,
                       timeout=300)
    assert r.returncode == 0, r.stderr
    out = json.loads(r.stdout.strip().splitlines()[-1])
    assert out["written back"] == out["put back"] == out["copied"] == out["new"], out
    assert out["named"] != out["new"], out
