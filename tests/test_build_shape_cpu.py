"""The shape of the neighbour build and its shared-memory limit, checked on the host.

tests/build_shape_check.cu calls the library's own build_group_shape, linked against stand-ins for
the CUDA runtime (tests/fake_cudart.cpp) that play a machine with three devices.  No GPU is needed."""
import os
import re
import shutil
import subprocess

import pytest

from paper_2003_14061_gb300 import build

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def shape(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("no nvcc")
    build.build()
    obj = os.path.join(build.BUILD, "kernels_rebuild.o")
    tmp = tmp_path_factory.mktemp("build_shape")
    if not os.path.exists(obj):
        obj = str(tmp / "kernels_rebuild.o")
        subprocess.run([nvcc, *build.ARCH, *build.FLAGS, "-c", os.path.join(build.CSRC, "kernels_rebuild.cu"), "-o", obj],
                       check=True)
    exe = str(tmp / "build_shape_check")
    subprocess.run([nvcc, *build.ARCH, *build.FLAGS, "-cudart", "none", os.path.join(HERE, "build_shape_check.cu"),
                    os.path.join(HERE, "fake_cudart.cpp"), obj, "-o", exe], check=True)

    def run(mode, cap, mean):
        out = subprocess.run([exe, str(mode), str(cap), str(mean)], capture_output=True, text=True, timeout=60, check=True)
        return {k: int(v) for k, v in re.findall(r"(\w+) (\d+)", out.stdout)}

    return run


@pytest.mark.parametrize("mode", [0, 1, 2])
@pytest.mark.parametrize("cap,mean", [(36, 11.8), (136, 77.6), (1000, 11.8), (4096, 300.0)])
def test_every_device_gets_the_limit(shape, mode, cap, mean):
    assert shape(mode, cap, mean)["bad"] == 0
