"""The g_h and udot solves give the same bits in every form they are run in:
the first sweep fused with its right-hand side or a kernel of its own
(CGL_OPT_UNFUSED_SWEEPS), over tiles of each of the three sizes, with all
fields in a block or one.  Precisions, bases, degrees and sweep counts."""
import numpy as np
import pytest

import inputs
from inputs import Mesh
from tests.test_gpu_parity import _problem, cgl  # noqa: F401

pytestmark = pytest.mark.gpu

# rows of elements of the strips: tiny tiles (float64), small, large
ROWS = (405, 1215, 10935)
KINDS = [(1, 0, 0), (1, 1, 0), (3, 0, 0), (3, 1, 0), (1, 0, 1), (3, 0, 1)]  # flux, precision, basis


def _state(flux, p, basis, seed, prec):
    mesh = Mesh(3, ROWS[0], p, 0.0, 3 / 8, 0.0, ROWS[0] / 8, basis=basis)
    make = inputs.random_euler_state if flux == 3 else inputs.random_scalar_state
    u = make(mesh, seed)
    return u.astype(np.float32).astype(np.float64) if prec else u


def _run(cgl, rows, flux, p, basis, prec, u, **prob):  # noqa: F811
    mesh = Mesh(3, rows, p, 0.0, 3 / 8, 0.0, rows / 8, basis=basis)
    st = cgl.State(cgl.Mesh(mesh), u.shape[0], prec)
    st.set_problem(dict(_problem(dict(flux=flux, mode=3, fl=1)).as_dict(), **prob))
    st.set_state(u)
    st.set_time(0.0)
    st.step(2)
    out = [st.get_state()] + [st.get_field(f) for f in (cgl.FIELD_GX, cgl.FIELD_GY, cgl.FIELD_R, cgl.FIELD_UDOT)]
    st.close()
    return [v.reshape(u.shape[0], -1, 3 * p) for v in out]


@pytest.mark.parametrize("kg,ku", [(1, 1), (2, 3), (0, 1), (3, 0)])
@pytest.mark.parametrize("p", [1, 2, 3, 4])
@pytest.mark.parametrize("flux,prec,basis", KINDS)
def test_fused_and_separate_sweeps(cgl, flux, prec, basis, p, kg, ku):  # noqa: F811
    u = _state(flux, p, basis, 17 + p, prec)
    for rows in ROWS[:1] if (kg, ku) != (2, 3) else ROWS:
        v = np.tile(u, (1, rows // ROWS[0], 1))
        a = _run(cgl, rows, flux, p, basis, prec, v, k_g=kg, k_u=ku)
        b = _run(cgl, rows, flux, p, basis, prec, v, k_g=kg, k_u=ku, options=cgl.OPT_UNFUSED_SWEEPS)
        for x, y in zip(a, b):
            assert np.array_equal(x, y), rows


@pytest.mark.parametrize("p", [1, 2, 3, 4])
@pytest.mark.parametrize("flux,prec,basis", KINDS)
def test_tile_sizes(cgl, flux, prec, basis, p):  # noqa: F811
    """A periodic strip repeated to the lengths of the other tile sizes steps like itself."""
    u = _state(flux, p, basis, 29 + p, prec)
    ref = None
    for rows in ROWS:
        n = rows // ROWS[0]
        out = _run(cgl, rows, flux, p, basis, prec, np.tile(u, (1, n, 1)), k_g=2, k_u=2)
        if ref is None:
            ref = out
        for x, y in zip(out, ref):
            assert np.array_equal(x, np.tile(y, (1, n, 1))), rows
