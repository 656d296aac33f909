"""A kept autotune choice decides only for the kernels that it was timed with: a line under a key of the grids alone,
as a build of other kernels left it, is not taken."""
import pytest

from paper_1904_10070_gb300 import vlb
from tests.test_gpu_ensemble import _members

pytestmark = pytest.mark.gpu


def _grids_key(count, ch_mode, grids, sms):
    x, mask = 1469598103934665603, (1 << 64) - 1
    for v in [count, ch_mode] + [n for g in grids for n in g]:
        for b in range(8):
            x = ((x ^ ((v >> (8 * b)) & 0xFF)) * 1099511628211) & mask
    return f"{x:016x}-{sms}"


def test_a_choice_of_other_kernels_is_not_taken(tmp_path, monkeypatch):
    import torch
    specs = [(28, 68, 2.1), (52, 124, 3.2)]
    mem = _members(specs, seed0=900)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    key = _grids_key(len(mem), mem[0][0]["ch_mode"], [(p["n_theta"], p["n_phi"]) for p, _ in mem], sms)
    cache = tmp_path / "tune.jsonl"
    cache.write_text(f'{{"key": "{key}", "kind": "ensemble", "sms": {sms}, "members": 2, "mode": 1, "tile_rows": 16, '
                     '"ctas_per_sm": 0, "ms": [99.0, 99.0, 99.0, 99.0]}\n')
    monkeypatch.setenv("VLB_AUTOTUNE_CACHE", str(cache))
    ens = vlb.Ensemble([vlb.make_params(**p, precision=vlb.FP32) for p, _ in mem])
    for v, (p, f) in zip(ens.views, mem):
        vlb.vlb_set_fields(v, f["rho"], f["ut"], f["up"], f["phi"])
    ens.step(2)
    ms = ens.config()["ms"]
    ens.close()
    assert max(ms) < 99.0
