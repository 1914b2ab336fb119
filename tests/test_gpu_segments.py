"""Tile lists at the lengths where the rasterisers cut them: one tile (d = 16)
that holds every Gaussian, so a list's length is the Gaussian count; the
segments are 256 entries in small calls and 512 in large ones, chunks of 32
and 64 entries inside them.  Held to the contract's tolerances (gemtest.py)."""
import numpy as np
import pytest
import torch

import gemtest as gt
import oracle
from paper_2509_25075_gb300 import synthetic as syn

pytestmark = pytest.mark.gpu


def _check(M, B, seed, tau=None):
    w = syn.Workload("seg", d=16, M=M, B=B, apix=1.2, n_clusters=1, s_lo=0.8, s_hi=3.0, seed=seed)
    tau = w.tau if tau is None else tau
    inp = gt.inputs(w)
    ctx = gt.context(w, tau=tau)
    args = [gt.to_dev(inp[k]) for k in ("params", "R", "t")]
    proj = torch.empty(B, 16, 16, device=gt.DEV)
    ctx.gem_project(*args, proj)
    ref = oracle.project(inp["params"], inp["R"], inp["t"], w.d, w.apix, tau)
    border = None if tau == 0 else gt.borderline_pairs(inp, w, tau) if M * B <= 20000 else np.full(B, 40)
    gt.assert_proj_close(proj.cpu().numpy(), ref, tau, border)
    again = torch.empty_like(proj)
    ctx.gem_project(*args, again)
    assert torch.equal(proj, again)
    g = syn.smooth_field(w) * 1e-3
    grad = torch.empty(M, 11, device=gt.DEV)
    ctx.gem_project_backward(gt.to_dev(g), grad)
    assert ctx.gem_status() == 0
    ref = oracle.grad(inp["params"], inp["R"], inp["t"], w.d, w.apix, tau, g)
    edge = oracle.grad_border(inp["params"], inp["R"], inp["t"], w.d, w.apix, tau, g, rel=1e-5) if tau else 0 * ref
    got = grad.cpu().numpy().astype(np.float64)
    assert np.linalg.norm(got - ref) <= 1e-4 * np.linalg.norm(ref) + np.linalg.norm(edge)
    ctx.close()


@pytest.mark.parametrize("M", [1, 31, 32, 33, 63, 64, 65, 127, 129, 255, 256, 257, 511, 513, 1023, 1025, 2100])
def test_list_lengths_in_a_small_call(M):
    _check(M, 2, seed=M)


@pytest.mark.parametrize("M", [1023, 1024, 1025, 2049])
def test_list_lengths_in_a_large_call(M):
    """About a million entries: the longest segments.  tau = 0, so that no pair
    is near the threshold."""
    _check(M, 1 + 1000000 // M, seed=M, tau=0.0)


@pytest.mark.parametrize("cfg", [0, 3, 7])
@pytest.mark.parametrize("B", [1, 151, 153, 1216, 1217, 2433, 3647, 3649, 5001])
def test_as_many_tasks_as_rounds_of_the_grid(B, cfg):
    """One task per image, around whole rounds of the grid (152 x 8, 5 and 1
    CTAs): every image is the bits it has in a call of seven views."""
    w = syn.Workload("task", d=16, M=40, B=7, apix=1.2, n_clusters=1, s_lo=0.8, s_hi=3.0, seed=5)
    inp = gt.inputs(w)
    params, R, t = (gt.to_dev(inp[k]) for k in ("params", "R", "t"))
    seven = torch.empty(7, 16, 16, device=gt.DEV)
    ctx = gt.context(w)
    ctx.gem_project(params, R, t, seven)
    ctx.close()
    view = torch.arange(B, device=gt.DEV) % 7
    ctx = gt.context(syn.Workload("task", d=16, M=40, B=B, apix=1.2, seed=5), tau=w.tau)
    ctx.gem_set_raster_config(cfg, -1)
    proj = torch.full((B, 16, 16), float("nan"), device=gt.DEV)
    for _ in range(2):
        ctx.gem_project(params, R[view].contiguous(), t[view].contiguous(), proj)
    assert ctx.gem_status() == 0
    assert float(seven.max()) > 0
    assert torch.equal(proj, seven[view])
    ctx.close()


@pytest.mark.parametrize("d,M,copies", [(16, 1500, 110), (16, 1500, 111), (16, 1500, 112), (64, 100, 103),
                                        (64, 100, 104), (64, 100, 105), (64, 100, 1)])
def test_backward_of_repeated_views(d, M, copies):
    """Calls on either side of the line between units of 128 and 256 entries
    (384 x 3040 entries), with few and with many entries per Gaussian and view
    (the two ways to add the moments): seven views over and over give the
    gradient of the seven, as often."""
    w = syn.Workload("rep", d=d, M=M, B=7, apix=1.2, n_clusters=1, s_lo=0.8, s_hi=3.0, seed=6)
    inp = gt.inputs(w)
    params, R, t = (gt.to_dev(inp[k]) for k in ("params", "R", "t"))
    g = gt.to_dev(syn.smooth_field(w) * 1e-3)
    grads = []
    for k in (1, copies):
        view = torch.arange(7 * k, device=gt.DEV) % 7
        ctx = gt.context(syn.Workload("rep", d=d, M=M, B=7 * k, apix=1.2, seed=6), tau=0.0,
                         max_pairs=7 * k * M * (d // 16) ** 2)
        proj = torch.empty(7 * k, d, d, device=gt.DEV)
        Rk, tk = R[view].contiguous(), t[view].contiguous()
        ctx.gem_project(params, Rk, tk, proj)
        grad = torch.empty(M, 11, device=gt.DEV)
        ctx.gem_project_backward(g[view].contiguous(), grad)
        assert ctx.gem_status() == 0
        assert ctx.gem_pair_count() == 7 * k * M * (d // 16) ** 2
        grads.append(grad.double())
        ctx.close()
    if copies == 1:  # the seven views themselves, against the oracle
        ref = oracle.grad(inp["params"], inp["R"], inp["t"], d, w.apix, 0.0, g.cpu().numpy())
        assert np.linalg.norm(grads[0].cpu().numpy() - ref) <= 1e-4 * np.linalg.norm(ref)
    err = float((grads[1] / copies - grads[0]).norm())
    assert err <= 1e-6 * float(grads[0].norm())
