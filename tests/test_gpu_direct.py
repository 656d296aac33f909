"""The direct stage kernel (FP64, WENO5, and FP32 grids off the packed layout) at the edges of its rules: one or
four threads per node (4864 nodes), partial tiles in both directions, rows of one to three columns whose
second and third neighbours wrap onto themselves, and WENO5 weights outside the range of the product form."""
import pytest

from paper_1904_10070_gb300 import vlb
from tests.test_gpu_parity import FP32_TOL, FP64_TOL, _compare, _random_fields

pytestmark = pytest.mark.gpu

GRIDS = [(76, 64), (77, 64), (9, 17), (8, 16), (64, 2), (129, 3), (4, 4099), (5, 33)]


@pytest.mark.parametrize("nt,ns", GRIDS)
@pytest.mark.parametrize("mode", [vlb.HYDRO, vlb.DIFFUSIVE])
@pytest.mark.parametrize("precision", [vlb.FP64, vlb.FP32])
def test_direct_stage_matches_the_oracle(nt, ns, mode, precision):
    p = dict(geometry=vlb.TORUS, R=2.3, r=1.0, n_theta=nt, n_phi=ns, dt=2e-3, tau=0.2, M=0.05, A=0.3, kappa=0.01,
             advection=vlb.UW3, ch_mode=mode)
    p["dt"] = min(2e-3, 0.5 * vlb.vlb_max_stable_dt(vlb.make_params(**p)))
    rho, ut, up, phi = _random_fields(nt, ns, seed=nt * 7919 + ns)
    _compare(p, rho, ut, up, phi, 6, precision, FP64_TOL if precision == vlb.FP64 else FP32_TOL)


@pytest.mark.parametrize("nt,ns,density", [(6, 2, 1.0), (6, 3, 1.0), (9, 33, 1.0), (16, 64, 1.0), (23, 95, 1.0),
                                           (16, 40, 1e6)])
@pytest.mark.parametrize("mode", [vlb.HYDRO, vlb.DIFFUSIVE])
@pytest.mark.parametrize("precision", [vlb.FP64, vlb.FP32])
def test_weno5_stage_matches_the_oracle(nt, ns, density, mode, precision):
    p = dict(geometry=vlb.TORUS, R=2.3, r=1.0, n_theta=nt, n_phi=ns, dt=2e-3, tau=0.2, M=0.05, A=0.3, kappa=0.01,
             advection=vlb.WENO5, ch_mode=mode)
    p["dt"] = min(2e-3, 0.5 * vlb.vlb_max_stable_dt(vlb.make_params(**p)))
    rho, ut, up, phi = _random_fields(nt, ns, seed=nt * 6007 + ns)
    _compare(p, density * rho, ut, up, phi, 3, precision, FP64_TOL if precision == vlb.FP64 else FP32_TOL)
