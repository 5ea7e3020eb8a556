"""Closed-loop runs into an output that is aligned for floats only, through the
C ABI: equal to those into an aligned one, nothing written beside them."""
import ctypes as C

import numpy as np
import pytest

from tests.gpu_util import need_gpu
from tests.test_slpv_gpu import _theta

pytestmark = pytest.mark.gpu
SC = np.array([20.0, 20.0, 2.0, 0.1, 0.1, 0.05], dtype=np.float32)


@pytest.mark.parametrize("nx,B,T", [(2, 1, 1), (4, 45, 9), (8, 33, 4), (4, 19500, 6)])
def test_output_of_any_float_alignment(nx, B, T):
    torch = need_gpu()
    from paper_2604_12505_gb300._lib import check, lib
    from paper_2604_12505_gb300.slpv import VelocityModel
    _, th = _theta(nx, 21, m1=0.2)
    rng = np.random.default_rng(B)
    F, tau, ref = (torch.tensor(a, device="cuda") for a in (rng.uniform(-20, 20, (B, T, 2)), rng.uniform(-2, 2, (B, T)),
                                                            rng.uniform(-0.3, 0.3, (B, T))))
    m = VelocityModel(nx=nx)
    m.set_params(th, SC)
    want = m.simulate(F, tau, ref, 0.05, 133.84, 0.2 * np.pi, 0.7).reshape(-1)
    for off in (1, 2, 3):
        buf = torch.full((B * T * 6 + 8,), 7.0, device="cuda")
        out = buf[off:off + B * T * 6]
        check(lib().slpv_simulate(m._h, B, T, C.c_void_p(F.data_ptr()), C.c_void_p(tau.data_ptr()),
                                  C.c_void_p(ref.data_ptr()), 0.05, 133.84, 0.2 * np.pi, 0.7,
                                  C.c_void_p(out.data_ptr()), torch.cuda.current_stream().cuda_stream))
        assert torch.equal(out, want)
        assert (buf[:off] == 7.0).all() and (buf[off + B * T * 6:] == 7.0).all()
    m.close()
