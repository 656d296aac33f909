"""The interface length of a diverged FP32 state.  An infinite high word of phi comes with a NaN low word: phi is NaN there,
and a NaN is on no side of 0, as in FP64."""
import numpy as np
import pytest

from paper_1904_10070_gb300 import vlb
from tests.gpu_helpers import gpu_params

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sign", [1.0, -1.0])
def test_a_diverged_phi_crosses_nothing(sign):
    import torch
    nt, ns = 8, 40
    p = dict(geometry=vlb.TORUS, R=2.3, r=1.0, n_theta=nt, n_phi=ns, dt=1e-4, tau=0.2, M=0.05, A=0.3, kappa=0.01,
             advection=vlb.UW3, ch_mode=vlb.HYDRO)
    z = np.zeros((nt, ns))
    s = vlb.Solver(gpu_params(p, vlb.FP32))
    s.set_fields(z + 1, z, z, z - sign * 0.5)
    ptr, stride = vlb.vlb_state_device(s.h)
    at = ptr - s.workspace.data_ptr()
    flat = s.workspace[at:at + 18 * stride * 4].view(torch.float32).view(18, stride)
    flat[16, 100] = sign * float("inf")
    flat[17, 100] = float("nan")
    torch.cuda.synchronize()
    assert s.interface_length() == 0.0
    s.close()
