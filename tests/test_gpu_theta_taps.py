"""The theta advection taps of the FP32 UW3 stages nearly cancel on a slowly varying population.  What their roundings
leave of the sum acts on the population itself, the same in every stage of a run: with four taps rounded to 2^-25 of
themselves (weights 1/6, 1, 1/2, 1/3 of v dt / h) it is some 1e-8 per stage at a Courant number of 0.4, which grows to about
2e-7 of the state over 64 steps; roundings at random leave about 1.3e-7.  Gate: 1.65e-7 between them, on the mean
over eight sets of axisymmetric fields against the FP64 stages, at tau = 0.1 where the advection dominates."""
import math

import numpy as np
import pytest

from oracle import vlb_oracle as O
from paper_1904_10070_gb300 import vlb
from tests.test_gpu_axisymmetric_drift import _fields

pytestmark = pytest.mark.gpu

GATE, STEPS, SEEDS = 1.65e-7, 64, 8


def _run(nt, ns, precision, fields):
    p = dict(geometry=vlb.TORUS, R=2.0, r=0.8, n_theta=nt, n_phi=ns, dt=1.0, tau=0.1, M=2.5e-3, A=0.5, kappa=5e-4,
             advection=vlb.UW3, ch_mode=vlb.HYDRO)
    ht, hp = p["r"] * 2.0 * math.pi / nt, (p["R"] - p["r"]) * 2.0 * math.pi / ns
    p["dt"] = 0.5 / (math.sqrt(3.0 + math.sqrt(6.0)) * (1.0 / ht + 1.0 / hp) + 0.5 / p["tau"])
    s = vlb.Solver(vlb.make_params(**p, precision=precision))
    s.set_fields(*[np.repeat(x, ns, axis=1) for x in fields])
    s.step(STEPS)
    f, _ = s.get_state()
    s.close()
    return f.reshape(4, 4, nt, ns)


@pytest.mark.parametrize("nt,ns", [(320, 40), (321, 41)])
def test_taps_cancel_as_a_whole(nt, ns):
    w, errs = O.weights(), []
    for seed in range(SEEDS):
        fields = _fields(77 + seed, nt)
        f32, f64 = _run(nt, ns, vlb.FP32, fields), _run(nt, ns, vlb.FP64, fields)
        norm = np.linalg.norm(f64 - f64.sum(axis=(0, 1)).mean() * np.outer(w, w)[:, :, None, None])
        errs.append(np.linalg.norm(f32 - f64) / norm)
    assert np.mean(errs) <= GATE, errs
