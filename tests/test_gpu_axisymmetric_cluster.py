"""Columns (n_phi = 1) on clusters of the portable size, which a device that refuses sixteen CTAs takes.  A row's
arithmetic does not depend on the CTA that owns it, so the bits are those of the larger cluster; the longest FP64 columns
fit eight CTAs only without the padding of their arrays."""
import numpy as np
import pytest

from paper_1904_10070_gb300 import vlb
from tests.test_gpu_parity import _random_fields

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nt", [320, 1000, 4080, 4081, 4096])
@pytest.mark.parametrize("adv", [vlb.UW3, vlb.WENO5])
@pytest.mark.parametrize("precision", [vlb.FP64, vlb.FP32])
def test_portable_cluster_gives_the_same_bits(nt, adv, precision):
    p = dict(geometry=vlb.TORUS, R=2.3, r=1.0, n_theta=nt, n_phi=1, dt=2e-3, tau=0.2, M=0.05, A=0.3, kappa=0.01,
             advection=adv, ch_mode=vlb.HYDRO)
    p["dt"] = min(2e-3, 0.5 * vlb.vlb_max_stable_dt(vlb.make_params(**p)))
    fields = _random_fields(nt, 1, seed=nt)
    states = []
    for route in (0, vlb.TEST_PORTABLE_CLUSTER):
        s = vlb.Solver(vlb.make_params(**p, precision=precision))
        vlb.vlb_test_route(s.h, route)
        s.set_fields(*fields)
        s.step(3)
        states.append(s.get_state())
        s.close()
    # four or sixteen threads share a row of an FP32 UW3 column, by its rows per CTA: not the same sums
    same_layout = precision == vlb.FP64 or adv == vlb.WENO5 or nt <= 240 or nt > 480
    for a, b in zip(*states):
        if same_layout:
            np.testing.assert_array_equal(a, b)
        else:
            np.testing.assert_allclose(a, b, rtol=0, atol=2e-5 * np.abs(a).max())
