"""The no-allocation step takes the same row table as a handle: both form its entries in FP64 and round them once, so that
one step from the same stored state gives the same bits on the packed FP32 grids (rows of coefficients
multiplied together in FP32 differ in about half of the entries).  A coefficient that host and device round to
different FP64 neighbours changes an FP32 entry about once in 2^28, so no difference is allowed for."""
import numpy as np
import pytest

from paper_1904_10070_gb300 import vlb
from tests.test_gpu_parity import _random_fields

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nt,ns,geom", [(48, 96, vlb.TORUS), (21, 44, vlb.TORUS), (160, 256, vlb.TORUS),
                                        (64, 64, vlb.FLAT)])
@pytest.mark.parametrize("mode", [vlb.HYDRO, vlb.DIFFUSIVE])
def test_one_step_gives_the_bits_of_the_handle(nt, ns, geom, mode):
    import torch
    p = dict(R=2.3, r=1.0, n_theta=nt, n_phi=ns, dt=1e-3, tau=0.2, M=0.05, A=0.3, kappa=0.01, geometry=geom,
             advection=vlb.UW3, ch_mode=mode)
    p["dt"] = min(1e-3, 0.5 * vlb.vlb_max_stable_dt(vlb.make_params(**p)))
    p = vlb.make_params(**p, precision=vlb.FP32)
    rho, ut, up, phi = _random_fields(nt, ns, seed=nt + ns)
    s = vlb.Solver(p)
    s.set_fields(rho, ut, up, phi)
    dA = 1.0 + (p.r / p.R if geom == vlb.TORUS else 0.0) * np.cos(np.arange(nt) * (2.0 * np.pi / nt))[:, None]
    m, e = np.frexp(float((dA * rho).sum() / (dA.sum() * ns)))
    n0 = float(np.ldexp(np.rint(np.ldexp(m, 20)), e - 20))  # the handle's reference density: 20 significant bits
    ptr, stride = vlb.vlb_state_device(s.h)
    at = ptr - s.workspace.data_ptr()
    view = s.workspace[at:at + 18 * stride * 4].view(torch.float32)
    state = view.clone()
    stream = torch.cuda.current_stream().cuda_stream
    vlb.vlb_step_noalloc(p, state.data_ptr(), stride, n0, 1, stream)
    s.step(1)
    a, b = (x.view(18, stride)[:, :nt * ns].cpu().numpy() for x in (state, view))
    s.close()
    np.testing.assert_array_equal(a, b)
