"""Totals and interface length where rows are cut into segments (few long rows): one segment and several, whole and
partial last passes, just below and above the number of rows that fill the launch.  Same gate as the other tests of
the totals: 1e-12 on the state read back."""
import numpy as np
import pytest

from oracle import vlb_oracle as O
from paper_1904_10070_gb300 import vlb
from tests.gpu_helpers import gpu_params, oracle_params

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nt,ns", [(4, 256), (4, 257), (5, 40001), (7, 5000), (256, 520), (257, 300), (1025, 31)])
@pytest.mark.parametrize("precision", [vlb.FP64, vlb.FP32])
def test_segments_cover_every_node_once(nt, ns, precision):
    p = dict(geometry=vlb.TORUS, R=2.3, r=1.0, n_theta=nt, n_phi=ns, dt=1e-4, tau=0.2, M=0.05, A=0.3, kappa=0.01,
             advection=vlb.UW3, ch_mode=vlb.HYDRO)
    rng = np.random.default_rng(nt * 131 + ns)
    s = vlb.Solver(gpu_params(p, precision))
    s.set_fields(1.0 + 0.1 * rng.uniform(-1, 1, (nt, ns)), *(0.05 * rng.uniform(-1, 1, (2, nt, ns))),
                 np.tanh(2.0 * rng.uniform(-1, 1, (nt, ns))))
    got, length = s.totals(), s.interface_length()
    f, ph = s.get_state()
    s.close()
    geo = O.Geometry(oracle_params(p))
    want = O.totals(f.reshape(4, 4, nt, ns), ph, geo)
    area = float(np.sum(np.broadcast_to(geo.dA, ph.shape)))
    for k, scale in enumerate((want[0], area, want[2], want[3])):
        assert abs(got[k] - want[k]) <= 1e-12 * scale, k
    ref = O.interface_length(ph, geo)
    assert abs(length - ref) <= 1e-12 * ref
