"""The FP32 stages over a few hundred launches against the FP64 ones: the momentum of the equilibrium balances that of
the populations.  With FP32 velocities sum w v v is 1 + 4.0e-8; uncorrected, the momentum grows by that times dt / tau in
every step, 64 x 0.84 x 4.0e-8 = 2.1e-6 here, where roundings of 2^-25 at random leave sqrt(192) x 2^-25 x a few, about
1e-6 times the share of the populations in them.  Gate: 8e-7 of the state's norm, for each of four sets of fields and
every FP32 UW3 kernel: packed pairs, grids off the packed layout, and the ragged members of an ensemble."""
import math

import numpy as np
import pytest

from oracle import vlb_oracle as O
from paper_1904_10070_gb300 import vlb

pytestmark = pytest.mark.gpu

GATE, STEPS = 8e-7, 64


def _smooth(rng, nt, ns, cells):
    x = rng.standard_normal((nt, ns))
    k2 = np.fft.fftfreq(nt)[:, None] ** 2 + np.fft.fftfreq(ns)[None, :] ** 2
    y = np.fft.ifft2(np.fft.fft2(x) * np.exp(-2.0 * (math.pi * cells) ** 2 * k2)).real
    y -= y.mean()
    return y / y.std()


def _fields(seed, nt, ns):
    rng = np.random.default_rng(seed)
    mean = rng.uniform(0.7, 1.4)
    return (mean * (1.0 + 0.005 * _smooth(rng, nt, ns, 4.0)), 0.03 * _smooth(rng, nt, ns, 4.0),
            0.03 * _smooth(rng, nt, ns, 4.0), np.tanh(2.5 * _smooth(rng, nt, ns, 3.0)))


def _params(nt, ns, adv, precision):
    p = dict(geometry=vlb.TORUS, R=2.0, r=0.8, n_theta=nt, n_phi=ns, dt=1.0, tau=2.5e-3, M=2.5e-3, A=0.5, kappa=5e-4,
             advection=adv, ch_mode=vlb.HYDRO)
    ht, hp = p["r"] * 2.0 * math.pi / nt, (p["R"] - p["r"]) * 2.0 * math.pi / ns
    p["dt"] = 0.5 / (math.sqrt(3.0 + math.sqrt(6.0)) * (1.0 / ht + 1.0 / hp) + 0.5 / p["tau"])
    return vlb.make_params(**p, precision=precision)


def _reference(nt, ns, adv, fields):
    s = vlb.Solver(_params(nt, ns, adv, vlb.FP64))
    s.set_fields(*fields)
    s.step(STEPS)
    f, _ = s.get_state()
    s.close()
    return f.reshape(4, 4, nt, ns)


def _check(f32, f64):
    v, w = O.velocities(), O.weights()
    norm = np.linalg.norm(f64 - f64.sum(axis=(0, 1)).mean() * np.outer(w, w)[:, :, None, None])
    for subs in ("ijqs,i->qs", "ijqs,j->qs"):
        drift = np.linalg.norm(np.einsum(subs, f32.reshape(f64.shape) - f64, v))
        assert drift <= GATE * norm, (subs, drift / norm)


@pytest.mark.parametrize("nt,ns,adv", [(40, 64, vlb.UW3), (41, 63, vlb.UW3)])
@pytest.mark.parametrize("seed", range(4))
def test_stage_momentum_does_not_drift(nt, ns, adv, seed):
    fields = _fields(seed, nt, ns)
    s = vlb.Solver(_params(nt, ns, adv, vlb.FP32))
    s.set_fields(*fields)
    s.step(STEPS)
    f, _ = s.get_state()
    s.close()
    _check(f, _reference(nt, ns, adv, fields))


def test_ensemble_momentum_does_not_drift():
    grids = [(40, 64), (41, 63), (37, 58)]
    fields = [_fields(10 + k, *g) for k, g in enumerate(grids)]
    ens = vlb.Ensemble([_params(*g, vlb.UW3, vlb.FP32) for g in grids])
    for v, f in zip(ens.views, fields):
        vlb.vlb_set_fields(v, *f)
    ens.step(STEPS)
    states = [vlb.vlb_get_state(v, *g)[0] for v, g in zip(ens.views, grids)]
    ens.close()
    for f, g, x in zip(states, grids, fields):
        _check(f, _reference(*g, vlb.UW3, x))
