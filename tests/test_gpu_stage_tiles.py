"""The packed FP32 stage at the edges of its tile rule (8 or 16 rows; 152 tiles of either height), with partial tiles
in both directions, and on grids below and just above one copy box."""
import pytest

from paper_1904_10070_gb300 import vlb
from tests.test_gpu_parity import FP32_TOL, _compare, _random_fields

pytestmark = pytest.mark.gpu

GRIDS = [(152, 256), (153, 256), (304, 252), (305, 256), (8, 32), (9, 36), (12, 40), (4868, 32), (17, 2436)]


def _params(nt, ns, mode):
    p = dict(geometry=vlb.TORUS, R=2.3, r=1.0, n_theta=nt, n_phi=ns, dt=2e-3, tau=0.2, M=0.05, A=0.3, kappa=0.01,
             advection=vlb.UW3, ch_mode=mode)
    p["dt"] = min(2e-3, 0.5 * vlb.vlb_max_stable_dt(vlb.make_params(**p)))
    return p


@pytest.mark.parametrize("nt,ns", GRIDS)
@pytest.mark.parametrize("mode", [vlb.HYDRO, vlb.DIFFUSIVE])
def test_stage_matches_the_oracle(nt, ns, mode):
    rho, ut, up, phi = _random_fields(nt, ns, seed=nt * 7919 + ns)
    _compare(_params(nt, ns, mode), rho, ut, up, phi, 3, vlb.FP32, FP32_TOL)
