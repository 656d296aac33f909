"""The structure-factor length where its sums run over hundreds of strips: each part is summed in FP64, the parts with
compensation, so that the length of a real coarsening field is as accurate as the FP64 FFT it is compared with
(a few units in the last place: 6e-16)."""
import numpy as np
import pytest

from oracle import vlb_oracle as O
from paper_1904_10070_gb300 import inputs, vlb
from tests.gpu_helpers import gpu_params, oracle_params

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nt,ns", [(64, 4096), (256, 2048), (1024, 1024)])
@pytest.mark.parametrize("seed", range(3))
def test_length_to_the_last_places(nt, ns, seed):
    p = dict(geometry=vlb.TORUS, R=2.3, r=1.0, n_theta=nt, n_phi=ns, dt=1e-5, tau=0.2, M=0.05, A=0.3, kappa=0.01,
             advection=vlb.UW3, ch_mode=vlb.HYDRO)
    phi = np.tanh(2.0 * inputs.noise(seed, nt, ns, 1.0) + np.cos(np.arange(nt) * (2.0 * np.pi / nt))[:, None])
    z = np.zeros((nt, ns))
    s = vlb.Solver(gpu_params(p, vlb.FP64))
    s.set_fields(z + 1.0, z, z, phi)
    got = s.structure_length()
    s.close()
    want = O.structure_length(phi, O.Geometry(oracle_params(p)))
    assert abs(got - want) <= 6e-16 * want
