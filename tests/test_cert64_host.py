"""The float32 certificate of the Euler limiters on float64 data: it must
never certify a factor whose float64 value differs from 1, also where density,
momentum, energy or the contributions leave the range of a float (host build of
the device code with nvcc; no GPU needed)."""
import json
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def check(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    exe = str(tmp_path_factory.mktemp("cert64") / "cert64_check")
    subprocess.run([nvcc, "-std=c++17", "-O2", "-o", exe, os.path.join(HERE, "native", "cert64_check.cu")],
                   check=True, capture_output=True)

    def run(*args):
        r = subprocess.run([exe, "300000", *map(str, args)], capture_output=True, text=True, check=True)
        return json.loads(r.stdout), r.stderr

    return run


# decades of the density and of m: ordinary ones (most factors are certified there), around and beyond
# the largest float, and where contributions or averages are subnormal or zero as floats
@pytest.mark.parametrize("decades,least", [((-8, 3, -9, -1), 0.2), ((30, 45, -9, -1), 0.0), ((37, 39, -2, 2), 0.0),
                                           ((38, 120, -20, 40), 0.0), ((20, 38, 0, 60), 0.0),
                                           ((-38, -30, -12, -1), 0.0), ((-45, -20, -30, -5), 0.0),
                                           ((-20, -5, -30, -1), 0.0), ((-8, 3, -40, -20), 0.0),
                                           ((-60, -20, 0, 40), 0.0)])
def test_certificate_on_float64_data(check, decades, least):
    out, err = check(*decades)
    assert out["wrong"] == 0, (out, err)
    assert out["certified"] >= least * out["trials"], out
