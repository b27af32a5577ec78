"""Meshes whose arrays of several values per element hold more than 2^31 of
them: the FP64 and FP32-mixed Euler stages keep 14 per element beside others.
A periodic state of 12700 x 12700 Q1 elements that repeats one of 100 x 127
must step bitwise like the small one (same element side, same time step)."""
import numpy as np
import pytest

import inputs
from inputs import Mesh
from tests.test_gpu_parity import _problem, cgl  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,gigabytes", [(1, 110), (0, 190)], ids=["mixed", "fp64"])
def test_more_values_than_32_bit_offsets(cgl, prec, gigabytes):  # noqa: F811
    import torch
    if torch.cuda.mem_get_info()[0] < gigabytes * 10 ** 9:
        pytest.skip("needs %d GB of free device memory" % gigabytes)
    nx, ny, N = 100, 127, 12700
    assert 14 * N * N > 2 ** 31 and N % nx == 0 and N % ny == 0
    prob = _problem(dict(flux=3, mode=3, fl=1))
    small = Mesh(nx, ny, 1, 0.0, nx / 128, 0.0, ny / 128)
    u0 = inputs.random_euler_state(small, 11)
    if prec:
        u0 = u0.astype(np.float32).astype(np.float64)
    st = cgl.State(cgl.Mesh(small), 4, cgl.FP32_MIXED if prec else cgl.FP64)
    st.set_problem(prob)
    st.set_state(u0)
    st.set_time(0.0)
    st.step(1)
    ref = torch.tensor(st.get_state(), dtype=torch.float32 if prec else torch.float64, device="cuda")
    st.close()
    u = torch.tensor(u0, dtype=ref.dtype, device="cuda").repeat(1, N // ny, N // nx)
    torch.cuda.synchronize()
    st = cgl.State(cgl.Mesh(Mesh(N, N, 1, 0.0, N / 128, 0.0, N / 128)), 4, cgl.FP32_MIXED if prec else cgl.FP64,
                   u_device=u.data_ptr(), u_bytes=u.numel() * u.element_size())
    st.set_problem(prob)
    st.set_time(0.0)
    st.step_async(1)
    c = st.counters()  # waits for the step
    assert c["violations"] == c["nonfinite"] == 0
    for r in range(N // ny):
        rows = u[:, r * ny:(r + 1) * ny].reshape(4, ny, N // nx, nx)
        assert bool((rows == ref[:, :, None, :]).all()), r
    st.close()
    del u, ref
    torch.cuda.empty_cache()
