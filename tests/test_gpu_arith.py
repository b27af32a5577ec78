"""The arithmetic routines of the kernels that stand for hardware or library
operations (common.cuh, modal.cuh), on the device: square roots and reciprocals
at zero, at subnormals, at the ends of the range and at infinity, and over the
normal range in units of the last place; and whole stages with values there."""
import json
import math
import os
import shutil
import subprocess

import numpy as np
import pytest

import inputs
from inputs import Mesh
import oracle.scheme as S
from tests.test_gpu_parity import TOL64, _problem, _rel, cgl  # noqa: F401

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def arith(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    exe = str(tmp_path_factory.mktemp("arith") / "arith_check")
    subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-std=c++17", "-O2",
                    "--expt-relaxed-constexpr", "-o", exe, os.path.join(HERE, "native", "arith_check.cu")],
                   check=True, capture_output=True)
    r = subprocess.run([exe], capture_output=True, text=True, check=True)
    return json.loads(r.stdout)


def _points(arith, name):
    return [(float.fromhex(x), float.fromhex(y)) for x, y in arith["points"][name]]


def test_square_root(arith):
    """Within one unit in the last place over the normal range (x y is rounded once, the correction
    halves that error, the last sum rounds once more); zeros, subnormals and infinity like sqrt."""
    assert arith["root_d"] <= 1.0
    for x, y in _points(arith, "root_d"):
        if x == 0.0 or math.isinf(x):
            assert y == x
        else:
            assert abs(y - math.sqrt(x)) <= 2.0 ** -52 * math.sqrt(x), (x, y)


def test_conversions(arith):
    """widen is exact, narrow cuts to 24 bits; split_ff's pair rounds the high part to nearest and the
    rest, 28 bits, to 24: half a unit of 2^-24 and 8 of 2^-53 of the value's power of two."""
    assert arith["widen"] == 0.0
    assert arith["narrow"] <= 1.0
    assert arith["split_hi"] <= 0.5
    assert arith["split_pair"] <= 8.0


@pytest.mark.parametrize("p,basis", [(1, 0), (2, 0), (3, 0), (4, 0), (2, 1)])
def test_float64_gas_at_rest_with_a_narrow_velocity_pulse(cgl, p, basis):  # noqa: F811
    """exp(-r^2 / s^2) passes through every scale down to the smallest subnormal: the squares of the
    speeds of 1.5e-162 to 1.5e-154 are subnormal, on a ring that is wider than an element here."""
    mesh = Mesh(96, 12, p, 0.0, 1.0, 0.0, 0.125, 1, 1, basis=basis)
    prob = _problem(dict(flux=3, mode=3, fl=1))
    X, Y = inputs.node_coords(mesh)
    r2 = ((X - 0.2) ** 2 + (Y - 0.06) ** 2) / 0.025 ** 2
    rho = 1.0 + 0.2 * np.sin(5.0 * X) * np.cos(9.0 * Y)
    vx, vy = 0.3 * np.exp(-r2), -0.2 * np.exp(-r2)
    u = np.stack([rho, rho * vx, rho * vy, 2.5 * (1.0 + 0.1 * np.cos(7.0 * X)) + 0.5 * rho * (vx * vx + vy * vy)])
    band = (np.hypot(vx, vy) > 2e-162) & (np.hypot(vx, vy) < 1e-154)
    assert band.sum() > 4 * (p + 1)
    om = S.OracleMesh(mesh)
    dt = 0.5 * S.time_step(om, prob, u)
    ref, info = S.ssp_stage(om, prob, u, u, dt, 0.0, 1.0)
    st = cgl.State(cgl.Mesh(mesh), 4, cgl.FP64)
    st.set_problem(prob)
    st.set_state(u)
    st.set_base_state(u)
    st.stage(dt, 0.0, 1.0)
    out, gam, nu = st.get_state(), st.get_field(cgl.FIELD_GAMMA), st.get_field(cgl.FIELD_NU)
    st.close()
    d = prob.as_dict()
    nu_ref = S.element_speed(om, om.blocks(u), d) * om.h / (2 * p)
    assert np.abs(nu - nu_ref).max() <= 1e-13 * nu_ref.max()
    assert np.abs(gam - S.sensor(om, om.blocks(u), d)).max() <= 1e-10
    assert _rel(out, ref, 4) <= TOL64


@pytest.mark.parametrize("name,least", [("recip_d", 2.0 ** -1074), ("recip_f", 2.0 ** -149)])
def test_reciprocal(arith, name, least):
    """Within one unit in the last place over the normal range; infinity at zero, zero at infinity."""
    assert arith[name] <= 1.0
    u = 2.0 ** (-52 if name == "recip_d" else -23)
    for x, y in _points(arith, name):
        if name == "recip_f":
            with np.errstate(over="ignore"):
                x = float(np.float32(x))
        if x == 0.0:
            assert y == math.inf
        elif math.isinf(x):
            assert y == 0.0
        elif 1.0 / x > 3.4e38 and name == "recip_f":
            assert y == math.inf
        else:
            assert y == 1.0 / x or abs(y - 1.0 / x) <= max(u / x, least), (x, y)


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("flux,p", [(1, 1), (1, 2), (2, 3), (1, 4), (3, 2)])
def test_flat_element_without_gamma_eps(cgl, flux, p, prec):  # noqa: F811
    """gamma_eps = 0: an element with constant coefficients among others that are not has the ratio
    num / 0 and so gamma = 0, full dissipation at the foot of a jump, in both precisions."""
    mesh = Mesh(9, 8, p, 0.0, 9 / 8, 0.0, 1.0)
    prob = _problem(dict(flux=flux, mode=3, fl=1, gamma_eps=0.0))
    make = inputs.random_euler_state if flux == 3 else (
        lambda m, s: inputs.random_scalar_state(m, s, prob.umin, prob.umax, 0.4))
    u = make(mesh, 5 + p).astype(np.float32).astype(np.float64)
    for c in range(u.shape[0]):
        u[c, 3 * p:4 * p + 1, 4 * p:5 * p + 1] = u[c, 3 * p, 4 * p]
    om = S.OracleMesh(mesh)
    with np.errstate(divide="ignore"):
        ref = S.sensor(om, om.blocks(u), prob.as_dict())
    assert ref[3 * 9 + 4] == 0.0
    st = cgl.State(cgl.Mesh(mesh), u.shape[0], prec)
    st.set_problem(prob)
    st.set_state(u)
    st.set_base_state(u)
    st.stage(1e-4, 0.0, 1.0, raise_on_idp=False)
    gam = st.get_field(cgl.FIELD_GAMMA)
    st.close()
    assert gam[3 * 9 + 4] == 0.0
    assert np.abs(gam - ref).max() <= (5e-6 if prec else 1e-10)
