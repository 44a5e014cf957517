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

    def run(mode, cap, mean, dense=17.7):
        out = subprocess.run([exe, str(mode), str(cap), str(mean), str(dense)], capture_output=True, text=True, timeout=60, check=True)
        return {k: int(v) for k, v in re.findall(r"(\w+) (\d+)", out.stdout)}

    return run


@pytest.mark.parametrize("mode", [0, 1, 2])
@pytest.mark.parametrize("cap,mean", [(36, 11.8), (136, 77.6), (1000, 11.8), (4096, 300.0)])
def test_every_device_gets_the_limit(shape, mode, cap, mean):
    assert shape(mode, cap, mean)["bad"] == 0


@pytest.mark.parametrize("mode", [0, 1])
@pytest.mark.parametrize("mean,dense", [(0.1, 17.7), (11.8, 17.7), (14.7, 17.7), (7.8, 110.3), (77.6, 110.3), (55.0, 748.0)])
def test_a_generous_capacity_costs_no_warps(shape, mode, mean, dense):
    # r_c + skin of 1.52 (WCA), 2.8 and 5.3, from thin gases to liquids: beyond what the densest liquid
    # needs, a larger capacity changes nothing
    enough = int(1.6 * dense + 24)
    want = shape(mode, enough, mean, dense)
    for cap in (enough + 4, 1300, 4096):
        got = shape(mode, cap, mean, dense)
        assert got["bad"] == 0 and got["warps"] == want["warps"] and abs(got["rows"] - want["rows"]) <= 1
    # up to there the lists follow the capacity: a slab around an atom of the dense liquid holds 69 %
    assert want["rows"] >= 0.69 * dense
    assert shape(mode, 36, 11.8)["warps"] == 32 and shape(mode, 136, 77.6, 110.3)["warps"] >= 24


def test_rows_follow_the_mean_where_it_needs_more(shape):
    for mean in (80.0, 150.0, 400.0, 2000.0):
        got = shape(1, 4000, mean, 17.7)
        assert got["rows"] >= min(0.69 * 1.35 * mean + 12, 0.9 * 3500) and got["warps"] >= 1
        assert got["smem"] <= 232448 - 2048
