"""The CTF step and the FSC at every supported side (the transforms are
instantiated one by one): prediction, adjoint and losses against torch.fft in
float64, and the FSC's shell sums."""
import numpy as np
import pytest
import torch

import gemtest as gt
from paper_2509_25075_gb300 import synthetic as syn

pytestmark = pytest.mark.gpu

SIDES = [16, 32, 48, 64, 96, 128, 144, 192, 256, 288, 384, 432, 512, 576, 768]


@pytest.mark.parametrize("d", SIDES)
def test_ctf_step(d):
    B = 2
    w = syn.Workload("fs", d=d, M=1, B=B, apix=1.2, seed=d)
    proj, imgs, arr = gt.to_dev(syn.smooth_field(w)), gt.to_dev(syn.images(w)), gt.to_dev(syn.ctf_array(w))
    ctx = gt.context(w)
    pred, dproj = torch.empty_like(proj), torch.empty_like(proj)
    li = torch.empty(B, dtype=torch.float64, device=gt.DEV)
    ctx.gem_ctf_loss(proj, imgs, ctf=arr, pred=pred, dproj=dproj, loss_img=li)
    H = torch.zeros(B, d, d, dtype=torch.float64, device=gt.DEV)
    neg = (-torch.arange(d, device=gt.DEV)) % d
    H[:, :, :d // 2 + 1] = arr.double()
    H[:, :, d // 2 + 1:] = arr.double()[:, neg][:, :, neg[d // 2 + 1:]]
    H = 0.5 * (H + H[:, neg][:, :, neg])
    ref = torch.fft.ifft2(H * torch.fft.fft2(proj.double())).real
    r = ref - imgs.double()
    g = torch.fft.ifft2(H * torch.fft.fft2(2 * r / (B * d * d))).real
    assert (pred.double() - ref).abs().max() <= 1e-5 * ref.abs().max()
    assert (dproj.double() - g).abs().max() <= 2e-6 * g.abs().max()
    assert torch.allclose(li, (r * r).mean((1, 2)), rtol=1e-5)
    ctx.close()


@pytest.mark.parametrize("d", [s for s in SIDES if s <= 288])
def test_fsc(d):
    g = torch.Generator(device="cuda").manual_seed(d)
    a = torch.randn(d, d, d, device=gt.DEV, generator=g)
    b = a + torch.randn(d, d, d, device=gt.DEV, generator=g)
    ctx = gt.context(syn.Workload("fs", d=d, M=1, B=1, apix=1.2, seed=1))
    _, sums, _ = ctx.gem_fsc(a, b)
    F1, F2 = torch.fft.fftn(a.double()), torch.fft.fftn(b.double())
    k = torch.fft.fftfreq(d, 1.0 / d, device=gt.DEV, dtype=torch.float64).round()
    shell = torch.floor((k[:, None, None] ** 2 + k[None, :, None] ** 2 + k[None, None, :] ** 2).sqrt() + 0.5).long()
    n = d // 2 + 1
    at = shell < n
    for i, x in enumerate(((F1 * F2.conj()).real, F1.abs() ** 2, F2.abs() ** 2)):
        ref = torch.bincount(shell[at], x[at], n)
        scale = torch.bincount(shell[at], (F1.abs() * F2.abs())[at], n)
        assert ((sums[i] - ref).abs() <= 2e-6 * torch.maximum(scale, ref.abs())).all()
    ctx.close()
