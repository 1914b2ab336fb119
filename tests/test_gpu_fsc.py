"""GPU parity of the Fourier shell correlation (Eq. fsc) through the C ABI
against the oracle: random and correlated maps on several grid sizes, maps
made by the density query, and the threshold crossing."""
import numpy as np
import pytest
import torch

import gemtest as gt
import oracle
from paper_2509_25075_gb300 import synthetic as syn

pytestmark = pytest.mark.gpu


def _ctx(d, apix=1.2):
    return gt.context(syn.Workload("fsc", d=d, M=16, B=1, apix=apix, seed=1))


def _compare(ctx, X1, X2, thr=0.143):
    fsc, sums, res = ctx.gem_fsc(gt.to_dev(X1), gt.to_dev(X2), thr)
    assert ctx.gem_status() == 0
    c, (num, p1, p2), r = oracle.fsc(X1.astype(np.float32), X2.astype(np.float32), ctx.apix, thr)
    got = sums.cpu().numpy()
    # sums: relative to the shell's power scale
    scale = np.sqrt(p1 * p2)
    np.testing.assert_allclose(got[1], p1, rtol=2e-5, atol=1e-6 * p1.max())
    np.testing.assert_allclose(got[2], p2, rtol=2e-5, atol=1e-6 * p2.max())
    assert np.all(np.abs(got[0] - num) <= 2e-5 * scale + 1e-6 * scale.max())
    np.testing.assert_allclose(fsc.cpu().numpy(), c, atol=5e-5)
    return float(res.item()), r, c


@pytest.mark.parametrize("d", [16, 48, 96])
def test_fsc_random_maps(d):
    rng = np.random.default_rng(d)
    X1 = rng.normal(size=(d, d, d)).astype(np.float32)
    X2 = (0.7 * X1 + 0.5 * rng.normal(size=(d, d, d))).astype(np.float32)
    _compare(_ctx(d), X1, X2)


def test_fsc_crossing_of_correlated_maps():
    """Two noisy copies of a smooth map: the FSC falls with frequency and
    crosses 0.143; the GPU crossing agrees with the oracle's."""
    d = 64
    rng = np.random.default_rng(80)
    k = np.fft.fftfreq(d)
    k2 = k[:, None, None] ** 2 + k[None, :, None] ** 2 + k[None, None, :] ** 2
    signal = np.real(np.fft.ifftn(np.fft.fftn(rng.normal(size=(d, d, d))) * np.exp(-k2 / (2 * 0.08 ** 2))))
    signal /= signal.std()
    X1 = (signal + 0.3 * rng.normal(size=(d, d, d))).astype(np.float32)
    X2 = (signal + 0.3 * rng.normal(size=(d, d, d))).astype(np.float32)
    ctx = _ctx(d, apix=1.3)
    res, r, c = _compare(ctx, X1, X2)
    assert c[1] > 0.9 and c[-1] < 0.143
    assert 2 * 1.3 < r < d * 1.3
    assert res == pytest.approx(r, rel=1e-4)


@pytest.mark.parametrize("name", ["A2", "A3"])
def test_fsc_of_query_maps(name):
    """Half-maps in the GSFSC sense: the density of the Gaussians and of a
    perturbed copy, both from the density query."""
    w = syn.WORKLOADS[name]
    th = syn.gaussians(w)
    rng = np.random.default_rng(81)
    th2 = th.copy()
    th2[:, 0:3] += rng.normal(scale=0.3 * w.apix, size=(w.M, 3)).astype(np.float32)
    ctx = gt.context(w)
    v1 = ctx.gem_query(gt.to_dev(th), w.tau_query).clone()
    v2 = ctx.gem_query(gt.to_dev(th2), w.tau_query).clone()
    X1, X2 = v1.cpu().numpy(), v2.cpu().numpy()
    res, r, _ = _compare(ctx, X1, X2)
    assert res == pytest.approx(r, rel=1e-4)


def test_fsc_rejects_bad_threshold():
    from paper_2509_25075_gb300 import binding
    ctx = _ctx(16)
    X = torch.zeros(16, 16, 16, device=gt.DEV)
    with pytest.raises(binding.GemError) as ei:
        ctx.gem_fsc(X, X, 1.5)
    assert ei.value.code == binding.GEM_EINVAL


@pytest.mark.parametrize("d", [384, 432, 512, 576, 768])
def test_fsc_large_sides(d):
    """The shell sums at the sides whose transforms take 8 lines per block and
    whose shell sums need more than 48 KB, against torch.fft in float64.  A
    float32 transform of n values is off by at most about 2^-24 log2 n of
    their rms (both maps share one complex transform), and a run of 32
    products by 2^-19 of their absolute sum."""
    g = torch.Generator(device="cuda").manual_seed(d)
    a = torch.randn(d, d, d, device=gt.DEV, generator=g)
    b = a + torch.randn(d, d, d, device=gt.DEV, generator=g)
    ctx = _ctx(d)
    _, sums, _ = ctx.gem_fsc(a, b)
    assert ctx.gem_status() == 0
    k = torch.fft.fftfreq(d, 1.0 / d, device=gt.DEV, dtype=torch.float64).round()
    k2 = k[:, None, None] ** 2 + k[None, :, None] ** 2 + k[None, None, :] ** 2
    shell = torch.floor(k2.sqrt() + 0.5).long()
    n = d // 2 + 1
    at = shell < n
    shell = shell[at]
    F1, F2 = (torch.fft.fftn(x.double())[at] for x in (a, b))
    total = lambda x: torch.bincount(shell, x, n)  # noqa: E731
    A1, A2 = F1.abs(), F2.abs()
    delta = 2.0 ** -24 * np.log2(float(d) ** 3) * float((A1 ** 2 + A2 ** 2).mean().sqrt())
    s1, s2 = total(A1), total(A2)
    for i, (ref, terms) in enumerate([((F1 * F2.conj()).real, delta * (s1 + s2)),
                                      (A1 ** 2, 2 * delta * s1), (A2 ** 2, 2 * delta * s2)]):
        allow = terms + 2.0 ** -19 * total(ref.abs())
        assert ((sums[i] - total(ref)).abs() <= allow).all()
    ctx.close()
