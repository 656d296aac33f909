"""The axisymmetric cluster kernels (n_phi = 1) at the edges of their rules: a single CTA, blocks of uneven
size, the two thread layouts (up to 30 rows a CTA or more), and columns too large for the row table."""
import pytest

from paper_1904_10070_gb300 import vlb
from tests.test_gpu_parity import FP32_TOL, FP64_TOL, _compare, _random_fields

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nt,adv", [(4, vlb.UW3), (7, vlb.UW3), (15, vlb.UW3), (17, vlb.UW3), (250, vlb.UW3),
                                    (480, vlb.UW3), (481, vlb.UW3), (4096, vlb.UW3), (6, vlb.WENO5), (29, vlb.WENO5),
                                    (4096, vlb.WENO5)])
@pytest.mark.parametrize("mode", [vlb.HYDRO, vlb.DIFFUSIVE])
@pytest.mark.parametrize("precision", [vlb.FP64, vlb.FP32])
def test_axisymmetric_column_matches_the_oracle(nt, adv, mode, precision):
    p = dict(geometry=vlb.TORUS, R=2.3, r=1.0, n_theta=nt, n_phi=1, dt=2e-3, tau=0.2, M=0.05, A=0.3, kappa=0.01,
             advection=adv, ch_mode=mode)
    p["dt"] = min(2e-3, 0.5 * vlb.vlb_max_stable_dt(vlb.make_params(**p)))
    rho, ut, up, phi = _random_fields(nt, 1, seed=nt * 104729)
    _compare(p, rho, ut, up, phi, 7, precision, FP64_TOL if precision == vlb.FP64 else FP32_TOL)
