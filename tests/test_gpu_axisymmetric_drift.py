"""The FP32 axisymmetric kernels over a few hundred stages and many sets of fields, against the oracle.

What a stage rounds at random grows with the root of the number of stages and is forgotten at the rate of the
relaxation; what it rounds the same way every time (a constant, a product that stays the same over a run) grows with
the number itself.  The momentum shows it: its balance of n u / tau against the sum of v g / tau, off by one part in
2^24, is off by 192 x 0.57 x 2^-24 = 6.5e-6 of the momentum after 64 steps at dt / tau = 0.57, while roundings of 2^-25
at random leave sqrt(192) x 2^-25 x a few = about 1e-6 times the share of the populations in them.  The gate is 8e-7 of
the state's norm, on every one of the sets: mean densities from 0.7 to 1.4 (another reference density, another
rounding of everything that it enters) and two time steps, on both thread layouts (320 and 500 rows)."""
import math

import numpy as np
import pytest

from oracle import vlb_oracle as O
from paper_1904_10070_gb300 import vlb
from tests.gpu_helpers import gpu_params, oracle_params

pytestmark = pytest.mark.gpu

GATE = 8e-7


def _smooth(rng, nt, cells):
    x = rng.standard_normal(nt)
    k = np.fft.fftfreq(nt)
    y = np.fft.ifft(np.fft.fft(x) * np.exp(-2.0 * (math.pi * cells) ** 2 * k * k)).real
    y -= y.mean()
    return (y / y.std())[:, None]


def _fields(seed, nt):
    rng = np.random.default_rng(seed)
    mean = rng.uniform(0.7, 1.4)
    return (mean * (1.0 + 0.005 * _smooth(rng, nt, 8.0)), 0.03 * _smooth(rng, nt, 10.0), 0.03 * _smooth(rng, nt, 10.0),
            np.tanh(2.5 * _smooth(rng, nt, 6.0)))


@pytest.mark.parametrize("nt", [320, 500])
@pytest.mark.parametrize("frac", [1.0, 0.83])
@pytest.mark.parametrize("seed", range(8))
def test_momentum_does_not_drift(nt, frac, seed):
    p = dict(geometry=vlb.TORUS, R=2.0, r=0.0025 * nt, n_theta=nt, n_phi=1, dt=1.0, tau=2.5e-3, M=2.5e-3, A=0.5, kappa=5e-4,
             advection=vlb.UW3, ch_mode=vlb.HYDRO)
    ht = p["r"] * 2.0 * math.pi / nt
    p["dt"] = frac * 0.5 / (math.sqrt(3.0 + math.sqrt(6.0)) / ht + 0.5 / p["tau"])
    rho, ut, up, phi = _fields(1000 * nt + seed, nt)
    s = vlb.Solver(gpu_params(p, vlb.FP32))
    s.set_fields(rho, ut, up, phi)
    s.step(64)
    f32, _ = s.get_state()
    s.close()
    f, ph = O.init_state(rho, ut, up, phi)
    f, ph = O.run(f, ph, O.Geometry(oracle_params(p)), 64)
    f, f32 = f.reshape(4, 4, nt), f32.reshape(4, 4, nt)
    v, w = O.velocities(), O.weights()
    norm = np.linalg.norm(f - f.sum(axis=(0, 1)).mean() * np.outer(w, w)[:, :, None])
    for axis in (0, 1):
        drift = np.einsum("ijq,i->q" if axis == 0 else "ijq,j->q", f32 - f, v)
        assert np.linalg.norm(drift) <= GATE * norm, (axis, np.linalg.norm(drift) / norm)
