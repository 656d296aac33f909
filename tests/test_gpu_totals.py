"""The conserved totals and the interface length against the oracle on the state read back: rows shorter and
longer than a CTA, a single column, and values outside the range of the FP32 kernel's float pairs (its FP64
path).  The state is the same on both sides, so the gate is the pairs' 2^-44 summed over a grid: 1e-12."""
import numpy as np
import pytest

from oracle import vlb_oracle as O
from paper_1904_10070_gb300 import vlb
from tests.gpu_helpers import gpu_params, oracle_params

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nt,ns", [(4, 1), (5, 3), (33, 257), (600, 130), (17, 1000)])
@pytest.mark.parametrize("scale", [1.0, 3e4])
@pytest.mark.parametrize("precision", [vlb.FP64, vlb.FP32])
def test_totals_and_interface_match_the_oracle(nt, ns, scale, precision):
    p = dict(geometry=vlb.TORUS, R=2.3, r=1.0, n_theta=nt, n_phi=ns, dt=1e-4, tau=0.2, M=0.05, A=0.3, kappa=0.01,
             advection=vlb.UW3, ch_mode=vlb.HYDRO)
    rng = np.random.default_rng(nt * 31 + ns)
    rho = 1.0 + 0.1 * rng.uniform(-1, 1, (nt, ns))
    ut, up = 0.05 * rng.uniform(-1, 1, (2, nt, ns))
    phi = np.tanh(2.0 * rng.uniform(-1, 1, (nt, ns)))
    phi[0, 0] *= scale
    phi[nt // 2, ns // 2] = 0.0
    s = vlb.Solver(gpu_params(p, precision))
    s.set_fields(rho, ut, up, phi)
    got, length = s.totals(), s.interface_length()
    f, ph = s.get_state()
    s.close()
    geo = O.Geometry(oracle_params(p))
    want = O.totals(f.reshape(4, 4, nt, ns), ph, geo)
    area = float(np.sum(np.broadcast_to(geo.dA, ph.shape)))
    assert abs(got[0] - want[0]) <= 1e-12 * want[0]
    assert abs(got[1] - want[1]) <= 1e-12 * area * np.max(np.abs(ph))
    assert abs(got[2] - want[2]) <= 1e-12 * want[2]
    assert abs(got[3] - want[3]) <= 1e-12 * want[3]
    ref = O.interface_length(ph, geo)
    assert abs(length - ref) <= 1e-12 * max(ref, 1.0)
