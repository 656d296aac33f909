"""A tall thin grid on the packed FP32 stage.  The launch has one row of blocks per tile row, and a grid dimension
holds 65535 of them: 524304 rows need 65538 tiles of 8 rows but only 32769 of 16, so the stage has to take
the taller tile.  The flat grid repeats a block of 48 rows, and so must its state: every repeat equals the first bit
for bit, and the first the 48-row grid of the same spacing within the FP32 tolerance of the parity tests (the two
round their row coefficients from different radii)."""
import numpy as np
import pytest

from paper_1904_10070_gb300 import vlb

pytestmark = pytest.mark.gpu

ROWS, COLS, BLOCK = 524304, 40, 48


def _state(s, nt):
    """The 16 population deviations and phi of a solver as device tensors [17][nt][COLS]."""
    import torch
    ptr, stride = vlb.vlb_state_device(s.h)
    at = ptr - s.workspace.data_ptr()
    flat = s.workspace[at:at + 17 * stride * 4].view(torch.float32)
    return flat.as_strided((17, nt, COLS), (stride, COLS, 1))


def _run(nt, r, fields):
    p = vlb.make_params(R=2.0, r=r, n_theta=nt, n_phi=COLS, dt=5e-4, tau=0.2, M=0.01, A=0.3, kappa=1e-3,
                        geometry=vlb.FLAT, precision=vlb.FP32)
    s = vlb.Solver(p)
    s.set_fields(*fields)
    s.step(2)
    return s


def test_tall_grid_steps_on_the_taller_tiles():
    import torch
    rng = np.random.default_rng(5)
    block = [1.0 + 0.1 * rng.uniform(-1, 1, (BLOCK, COLS)), 0.05 * rng.uniform(-1, 1, (BLOCK, COLS)),
             0.05 * rng.uniform(-1, 1, (BLOCK, COLS)), np.tanh(2.0 * rng.uniform(-1, 1, (BLOCK, COLS)))]
    small = _run(BLOCK, 1.0, block)
    want = _state(small, BLOCK).to(torch.float64)
    tall = _run(ROWS, ROWS / BLOCK, [np.tile(x, (ROWS // BLOCK, 1)) for x in block])
    got = _state(tall, ROWS).view(17, ROWS // BLOCK, BLOCK, COLS)
    assert torch.equal(got, got[:, :1].expand_as(got))
    got = got[:, 0].to(torch.float64)
    err = (got - want).flatten(1).norm(dim=1) / want.flatten(1).norm(dim=1).clamp_min(1e-3 * (BLOCK * COLS) ** 0.5)
    assert float(err.max()) <= 2e-5
    small.close()
    tall.close()
