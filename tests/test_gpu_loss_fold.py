"""Losses folded by the last blocks of the CTF step: at image counts around the
warps' and blocks' strides, with and without the per-image output, and again
on a second call (the counters are back at zero)."""
import pytest
import torch

import gemtest as gt
from paper_2509_25075_gb300 import binding

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d", [16, 48])
@pytest.mark.parametrize("B", [1, 2, 31, 33, 255, 257, 600])
def test_losses(d, B):
    g = torch.Generator(device=gt.DEV).manual_seed(B)
    proj = torch.randn(B, d, d, device=gt.DEV, generator=g)
    im = torch.randn(B, d, d, device=gt.DEV, generator=g)
    ctf = 2 * torch.rand(B, d, d // 2 + 1, device=gt.DEV, generator=g) - 1
    ctx = binding.Context(d, 1.0, B, 1)
    pred = torch.empty_like(proj)
    li, loss = (torch.empty(n, dtype=torch.float64, device=gt.DEV) for n in (B, 1))
    got = []
    for _ in range(2):
        ctx.gem_ctf_loss(proj, im, ctf=ctf, pred=pred, loss_img=li, loss=loss)
        got.append((li.clone(), loss.clone()))
        ctx.gem_ctf_loss(proj, im, ctf=ctf, loss=loss)
        got.append((li.clone(), loss.clone()))
    ctx.close()
    for a, b in got[1:]:
        assert torch.equal(a, got[0][0]) and torch.equal(b, got[0][1])
    # Parseval in float32: a few dozen roundings of 6e-8 on each term
    want = ((pred.double() - im.double()) ** 2).mean(dim=(1, 2))
    assert ((li - want).abs() <= 5e-6 * want).all()
    assert abs(loss.item() - li.mean().item()) <= 1e-13 * abs(loss.item())
