"""The totals of FP32 states where the float pairs of their kernel reach their limits: flows so slow that |u|^2 loses
bits or underflows, a phase so pure that 1 - phi^2 does, and few long rows.  The state is read
back, so both sides see the same numbers; the sums are compared with extended precision at what FP64 arithmetic
leaves of them: 1e-15 for max |u| and the mass, 1e-13 for Psi (FP64 forms 1 - phi^2 to 1e-16 of 1) where phi is not
within 1e-3 of 1."""
import numpy as np
import pytest

from oracle import vlb_oracle as O
from paper_1904_10070_gb300 import vlb
from tests.gpu_helpers import gpu_params, oracle_params

pytestmark = pytest.mark.gpu

L = np.longdouble


def _params(nt, ns, **kw):
    return {**dict(geometry=vlb.TORUS, R=2.3, r=1.0, n_theta=nt, n_phi=ns, dt=1e-4, tau=0.2, M=0.05, A=0.3, kappa=0.01,
                   advection=vlb.UW3, ch_mode=vlb.HYDRO), **kw}


def _device_state(s):
    """(16 population deviations, phi) of an FP32 solver in extended precision."""
    import torch
    ptr, stride = vlb.vlb_state_device(s.h)
    nt, ns = s.shape
    at = ptr - s.workspace.data_ptr()
    flat = s.workspace[at:at + 18 * stride * 4].view(torch.float32).view(18, stride)[:, :nt * ns].cpu().numpy()
    return flat[:16].astype(L).reshape(4, 4, nt, ns), (flat[16].astype(L) + flat[17]).reshape(nt, ns)


def _want(p, g, phi, n0):
    """(mass, phi total, Psi, max |u|) in extended precision."""
    geo = O.Geometry(oracle_params(p))
    v = O.velocities().astype(L)
    n = n0 + g.sum(axis=(0, 1))
    ut, up = np.einsum("ijqs,i->qs", g, v) / n, np.einsum("ijqs,j->qs", g, v) / n
    dA = np.broadcast_to(geo.dA, phi.shape).astype(L)
    dth, dph = 2 * L(np.pi) / p["n_theta"], 2 * L(np.pi) / p["n_phi"]
    J = (1 + L(p["r"]) / L(p["R"]) * np.cos(np.arange(p["n_theta"]) * dth))[:, None]
    g1 = (np.roll(phi, -1, 0) - np.roll(phi, 1, 0)) / (2 * L(p["r"]) * dth)
    g2 = (np.roll(phi, -1, 1) - np.roll(phi, 1, 1)) / (2 * L(p["R"]) * J * dph)
    psi = L(p["A"]) / 4 * ((1 - phi) * (1 + phi)) ** 2 + L(p["kappa"]) / 2 * (g1 * g1 + g2 * g2)
    return (n * dA).sum(), (phi * dA).sum(), (psi * dA).sum(), np.sqrt(ut * ut + up * up).max(), (abs(phi) * dA).sum()


def _solver(p, rho, ut, up, phi):
    s = vlb.Solver(gpu_params(p, vlb.FP32))
    s.set_fields(rho, ut, up, phi)
    return s


@pytest.mark.parametrize("speed", [1e-12, 1e-18, 1e-24, 1e-30])
def test_slow_flows_are_reported(speed):
    nt, ns = 33, 130
    p = _params(nt, ns)
    rng = np.random.default_rng(3)
    one = np.ones((nt, ns))
    s = _solver(p, one, speed * rng.uniform(-1, 1, (nt, ns)), speed * rng.uniform(-1, 1, (nt, ns)), 0.1 * one)
    g, phi = _device_state(s)
    want, got = _want(p, g, phi, L(1)), s.totals()
    s.close()
    assert 0 < want[3] < 2 * speed
    assert abs(got[3] - want[3]) <= 1e-15 * want[3]
    assert abs(got[0] - want[0]) <= 1e-15 * want[0]


@pytest.mark.parametrize("nt,ns", [(6, 40), (33, 257), (600, 130), (4, 20000)])
def test_totals_are_as_accurate_as_in_fp64(nt, ns):
    p = _params(nt, ns)
    rng = np.random.default_rng(nt + ns)
    rho = 1.0 + 0.1 * rng.uniform(-1, 1, (nt, ns))
    s = _solver(p, rho, *(0.05 * rng.uniform(-1, 1, (2, nt, ns))), np.tanh(2.0 * rng.uniform(-1, 1, (nt, ns))))
    g, phi = _device_state(s)
    geo = O.Geometry(oracle_params(p))
    dA = np.broadcast_to(geo.dA, rho.shape)
    n0 = float((dA * rho).sum() / dA.sum())  # the solver keeps 20 significant bits
    m, e = np.frexp(n0)
    want, got = _want(p, g, phi, L(np.ldexp(np.rint(np.ldexp(m, 20)), e - 20))), s.totals()
    s.close()
    assert abs(got[0] - want[0]) <= 2e-15 * want[0]
    assert abs(got[1] - want[1]) <= 2e-15 * want[4]
    assert abs(got[2] - want[2]) <= 2e-15 * want[2]
    assert abs(got[3] - want[3]) <= 1e-15 * want[3]


@pytest.mark.parametrize("off", [1e-3, 1e-6])
def test_free_energy_of_a_nearly_pure_phase(off):
    nt, ns = 40, 96
    p = _params(nt, ns, kappa=1e-30)
    rng = np.random.default_rng(9)
    one = np.ones((nt, ns))
    s = _solver(p, one, 0 * one, 0 * one, 1.0 - off * rng.uniform(0.5, 1.0, (nt, ns)))
    g, phi = _device_state(s)
    want, got = _want(p, g, phi, L(1)), s.totals()
    s.close()
    assert abs(got[2] - want[2]) <= 1e-13 * want[2]

