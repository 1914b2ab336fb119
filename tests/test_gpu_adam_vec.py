"""The optimiser step takes four entries per thread when every array is
16-byte aligned and one when not: the same bits either way, at entry counts
with every remainder of four, and with an imposed scale."""
import pytest
import torch

import gemtest as gt
from paper_2509_25075_gb300 import synthetic as syn

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("iso", [False, True])
@pytest.mark.parametrize("M", [1, 2, 3, 4, 5, 93, 94, 1000, 28299, 28300, 28301, 28303])
def test_aligned_and_unaligned_arrays_give_the_same_step(M, iso):
    ctx = gt.context(syn.Workload("av", d=16, M=M, B=1, seed=1))
    g = torch.Generator(device="cuda").manual_seed(M)
    src = [torch.randn(M, 11, device=gt.DEV, generator=g) * s for s in (1.0, 0.1, 0.0, 0.3)]
    src[2] = torch.rand(M, 11, device=gt.DEV, generator=g)
    src[3][0, 0] = float("nan")  # counts as a zero gradient
    scale = torch.rand(M, device=gt.DEV, generator=g) + 0.5 if iso else None
    out = {}
    for off in (0, 1):  # floats from a 16-byte boundary
        arrs = []
        for x in src + [torch.full((M, 11), -7.0, device=gt.DEV)]:
            y = torch.empty(11 * M + 4, device=gt.DEV)[off:off + 11 * M].view(M, 11)
            y.copy_(x)
            arrs.append(y)
        raw, m, v, grad, params = arrs
        ctx.gem_adam_step(raw, m, v, grad, params, (0.05, 0.01, 0.002, 0.02), 3, iso_scale=scale)
        out[off] = [raw, m, v, params]
    assert ctx.gem_status() == 0
    for a, b in zip(out[0], out[1]):
        assert torch.equal(a, b)
        assert not torch.isnan(a).any()
    ctx.close()
