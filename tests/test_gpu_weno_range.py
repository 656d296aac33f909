"""FP64 WENO5 weights outside the range of the product form, where the direct kernel forms a tile again with the plain
formula: the weights grow as the eighth power of the differences, so the rerun starts near differences of 1e31.  All
tiles of a grid, and one density peak that takes one tile of many out of range while its neighbours keep the
product form, against the oracle at the FP64 tolerance of the parity tests."""
import numpy as np
import pytest

from paper_1904_10070_gb300 import vlb
from tests.test_gpu_parity import FP64_TOL, _compare, _random_fields

pytestmark = pytest.mark.gpu


def _params(nt, ns, mode):
    p = dict(geometry=vlb.TORUS, R=2.3, r=1.0, n_theta=nt, n_phi=ns, dt=2e-3, tau=0.2, M=0.05, A=0.3, kappa=0.01,
             advection=vlb.WENO5, ch_mode=mode)
    p["dt"] = min(2e-3, 0.5 * vlb.vlb_max_stable_dt(vlb.make_params(**p)))
    return p


@pytest.mark.parametrize("nt,ns", [(16, 40), (9, 33)])
@pytest.mark.parametrize("mode", [vlb.HYDRO, vlb.DIFFUSIVE])
def test_every_tile_out_of_range(nt, ns, mode):
    rho, ut, up, phi = _random_fields(nt, ns, seed=nt * 6007 + ns)
    _compare(_params(nt, ns, mode), 1e34 * rho, ut, up, phi, 3, vlb.FP64, FP64_TOL)


@pytest.mark.parametrize("mode", [vlb.HYDRO, vlb.DIFFUSIVE])
@pytest.mark.parametrize("at", [(21, 70), (0, 0), (23, 95)])
def test_one_tile_out_of_range(mode, at):
    nt, ns = 24, 96
    rho, ut, up, phi = _random_fields(nt, ns, seed=11)
    q, s = np.arange(nt)[:, None] - at[0], np.arange(ns)[None, :] - at[1]
    q, s = (q + nt // 2) % nt - nt // 2, (s + ns // 2) % ns - ns // 2
    rho = 1e30 * rho * (1.0 + 300.0 * np.exp(-2.0 * (q * q + s * s)))
    _compare(_params(nt, ns, mode), rho, ut, up, phi, 2, vlb.FP64, FP64_TOL)
