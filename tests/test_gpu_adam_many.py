"""One Adam launch over many tensors against one launch each: the same bits, over sizes around a block, empty bf16
copies, and more tensors than one launch holds."""
import pytest

from paper_1904_10070_gb300 import vlb

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sizes", [[1], [255, 256, 257], [64, 9216, 36864, 16], [700000], [33] * 65])
def test_many_tensors_match_single_steps(sizes):
    import torch
    gen = torch.Generator(device="cuda").manual_seed(len(sizes))
    st = torch.cuda.current_stream().cuda_stream
    p, g, m, v = ([torch.rand(n, generator=gen, device="cuda") - (0.0 if sq else 0.5) for n in sizes]
                  for sq in (False, False, False, True))
    pb = [torch.zeros(n, dtype=torch.bfloat16, device="cuda") if k % 2 == 0 else None for k, n in enumerate(sizes)]
    ref = [[t.clone() if t is not None else None for t in ts] for ts in (p, g, m, v, pb)]
    for k, n in enumerate(sizes):
        vlb.vlb_adam_step(n, ref[0][k], ref[1][k], ref[2][k], ref[3][k], 7, 1e-3, 0.9, 0.999, 1e-8, ref[4][k], st)
    vlb.vlb_adam_step_many(p, g, m, v, 7, 1e-3, 0.9, 0.999, 1e-8, pb, st)
    for got, want in zip((p, g, m, v, pb), ref):
        for a, b in zip(got, want):
            assert (a is None and b is None) or torch.equal(a, b)
    with pytest.raises(vlb.VlbError):
        vlb.vlb_adam_step_many(p[:1], g[:1], m[:1], v[:1], 0, 1e-3, 0.9, 0.999, 1e-8, pb[:1], st)
