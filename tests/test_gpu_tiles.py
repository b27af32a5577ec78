"""Edges of the tiles of the stage kernels, against the FP64 oracle.

The g_h and udot stencils work on tiles of one of three sizes (up to 32 x 16
elements), the sensor and a scalar's low-order part on tiles of 32 x 8, 4 or 1
elements, the facets of systems on tiles of 32 x 4, the residual and the
update of systems on rows of 32.  The meshes are one tile and a remainder, or
narrow strips that are just long enough for the next tile size, so that the
large tiles are met with a small oracle.  Bounds: those of the stage parity
tests (float64 1e-12 of a component's magnitude; FP32-mixed 2e-6)."""
import numpy as np
import pytest

import inputs
from inputs import Mesh
import oracle.scheme as S
from tests.test_gpu_parity import TOL64, _case_state, _gpu_stage, _inward_f32, _problem, _rel, cgl  # noqa: F401

pytestmark = pytest.mark.gpu

SCALAR = dict(flux=1, mode=3, fl=1)
EULER = dict(flux=3, mode=3, fl=1)
# (nx, ny, p, bc_x, bc_y, problem): boundary conditions 0 periodic, 1 outflow, 2 fixed
SHAPES = [
    (33, 17, 1, 0, 0, dict(SCALAR, k_g=2, k_u=2)),
    (32, 16, 2, 0, 0, dict(SCALAR, k_g=1, k_u=0)),
    (31, 9, 2, 1, 0, dict(SCALAR, k_g=0, k_u=2)),
    (17, 13, 3, 0, 2, dict(SCALAR, k_g=2, k_u=1)),
    (9, 7, 4, 2, 0, dict(SCALAR, k_g=1, k_u=1)),
    (2, 3, 2, 0, 0, dict(SCALAR, k_g=2, k_u=2)),
    # the small tiles of float64: 152 or more of 8 or 6 rows of elements
    (3, 1217, 2, 0, 1, dict(SCALAR)),
    (3, 1217, 3, 0, 0, dict(SCALAR)),
    (3, 1217, 4, 2, 0, dict(SCALAR)),
    # the large tiles: 608 of 16 rows (p <= 2), 304 of 8 to 16
    (3, 9729, 1, 0, 0, dict(SCALAR, k_g=1, k_u=1)),
    (3, 9729, 2, 0, 2, dict(SCALAR, k_g=2, k_u=2)),
    (19457, 2, 2, 1, 0, dict(SCALAR)),
    (3, 4865, 3, 0, 0, dict(SCALAR)),
    (3, 3649, 4, 1, 1, dict(SCALAR)),
    # systems: rows of 32 elements and facet tiles of 32 x 4
    (1, 1, 2, 0, 0, dict(EULER)),
    (32, 4, 1, 1, 1, dict(EULER)),
    (33, 5, 2, 0, 0, dict(EULER)),
    (31, 3, 3, 1, 0, dict(EULER)),
    (65, 9, 2, 0, 1, dict(EULER)),
    (33, 8, 4, 0, 0, dict(EULER)),
    (3, 9729, 2, 0, 0, dict(EULER)),
    (33, 5, 2, 1, 1, dict(EULER, fl=0)),
    (33, 5, 2, 0, 1, dict(EULER, mode=0, fl=2)),
]


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "%s_%dx%d_p%d" % ("euler" if s[5]["flux"] == 3 else "burgers", *s[:3]))
def test_stage_at_tile_edges(cgl, shape, prec):  # noqa: F811
    nx, ny, p, bx, by, over = shape
    mesh = Mesh(nx, ny, p, 0.0, nx / 8, 0.0, ny / 8, bx, by)
    prob = _problem(over)
    u, un = _case_state(mesh, prob, 31 * nx + ny + p)
    if prec:
        u, un = (v.astype(np.float32).astype(np.float64) for v in (u, un))
        if prob.flux != inputs.FLUX_EULER:
            lo32, hi32 = _inward_f32(prob.umin, prob.umax)
            u, un = np.clip(u, lo32, hi32), np.clip(un, lo32, hi32)
    om = S.OracleMesh(mesh)
    dt = 0.5 * S.time_step(om, prob, u)
    ref, info = S.ssp_stage(om, prob, u, un, dt, 0.75, 0.25)
    out, ginfo, f = _gpu_stage(cgl, mesh, prob, u, un, dt, 0.75, 0.25, prec=prec)
    nc = u.shape[0]
    assert _rel(out, ref, nc) <= (2e-6 if prec else TOL64)
    assert _rel(f["ue"], info["ue"], nc) <= (1e-13 if prec else 1e-14)
    assert np.abs(f["dte"] - info["dte"]).max() <= (2e-6 if prec else 1e-13) * info["dte"].max()
    assert _rel(f["ubL"], info["ubL"], nc) <= (2e-6 if prec else 1e-13)
    assert _rel(f["ube"], info["ube"], nc) <= (5e-6 if prec else TOL64)
    if prob.mode != inputs.MODE_LO:
        assert np.abs(f["gamma"] - info["gamma"]).max() <= (5e-6 if prec else 1e-10)
    assert np.abs(f["beta"] - info["beta"]).max() <= (5e-5 if prec else 1e-10)
    assert ginfo["violations"] == info["violations"] == 0


@pytest.mark.parametrize("p", [1, 2, 3, 4])
def test_float64_limiter_option_changes_no_bit(cgl, p):  # noqa: F811
    """Systems in float64: the limiters' certificates (the positivity one
    evaluates its float32 form from float64 data) skip the exact formulas
    only where these give the same result."""
    mesh = Mesh(33, 9, p, 0.0, 33 / 9, 0.0, 1.0)
    prob = _problem(EULER)
    u, _ = _case_state(mesh, prob, 77 + p)
    out = []
    for opts in (0, cgl.OPT_FP64_LIMITER):
        st = cgl.State(cgl.Mesh(mesh), 4, cgl.FP64)
        st.set_problem(dict(prob.as_dict(), options=opts))
        st.set_state(u)
        st.step(3)
        out.append((st.get_state(), st.get_field(cgl.FIELD_BETA)))
        st.close()
    for a, b in zip(*out):
        assert np.array_equal(a, b)
