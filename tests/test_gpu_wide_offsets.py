"""FP64 stages with 64-bit offsets, which grids of 2^29 nodes and more take, against the 32-bit ones on the same tiles:
the same arithmetic, so the same bits; partial tiles in both directions and odd rows."""
import numpy as np
import pytest

from paper_1904_10070_gb300 import vlb
from tests.test_gpu_parity import _random_fields

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nt,ns", [(77, 64), (129, 41)])
@pytest.mark.parametrize("adv", [vlb.UW3, vlb.WENO5])
@pytest.mark.parametrize("mode", [vlb.HYDRO, vlb.DIFFUSIVE])
def test_wide_offsets_give_the_same_bits(nt, ns, adv, mode):
    p = dict(geometry=vlb.TORUS, R=2.3, r=1.0, n_theta=nt, n_phi=ns, dt=2e-3, tau=0.2, M=0.05, A=0.3, kappa=0.01,
             advection=adv, ch_mode=mode)
    p["dt"] = min(2e-3, 0.5 * vlb.vlb_max_stable_dt(vlb.make_params(**p)))
    fields = _random_fields(nt, ns, seed=nt * 31 + ns)
    states = []
    for route in (0, vlb.TEST_WIDE_OFFSETS):
        s = vlb.Solver(vlb.make_params(**p, precision=vlb.FP64))
        vlb.vlb_test_route(s.h, route)
        s.set_fields(*fields)
        s.step(3)
        states.append(s.get_state())
        s.close()
    for a, b in zip(*states):
        np.testing.assert_array_equal(a, b)
