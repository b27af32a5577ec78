"""A step whose launches are refused (a mesh with more rows of nodes than a
grid has rows of blocks) reports the error, leaves the state as it was and
leaves nothing behind for the next call of another state."""
import numpy as np
import pytest

import inputs
from inputs import Mesh
from tests.test_gpu_parity import _problem, cgl  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("flux", [1, 3])
@pytest.mark.parametrize("prec", [0, 1])
def test_refused_launch(cgl, flux, prec):  # noqa: F811
    make = inputs.random_euler_state if flux == 3 else inputs.random_scalar_state
    prob = _problem(dict(flux=flux, mode=3, fl=1))
    good, tall = Mesh(8, 8, 2), Mesh(2, 70000, 1, 0.0, 2 / 8, 0.0, 70000 / 8)
    ref = None
    for broken in (False, True):
        if broken:
            v = make(tall, 3).astype(np.float32).astype(np.float64)
            st = cgl.State(cgl.Mesh(tall), v.shape[0], prec)
            st.set_problem(prob)
            st.set_state(v)
            for call in (lambda: st.step(1), lambda: st.step_async(1), lambda: st.stage(1e-4, 0.0, 1.0)):
                with pytest.raises(cgl.CglError):
                    call()
            assert np.array_equal(st.get_state(), v)
            assert st.get_time() == 0.0
            st.close()
        u = make(good, 5)
        st = cgl.State(cgl.Mesh(good), u.shape[0], prec)
        st.set_problem(prob)
        st.set_state(u)
        st.step(2)
        out = st.get_state()
        st.close()
        if ref is None:
            ref = out
        assert np.array_equal(out, ref)
