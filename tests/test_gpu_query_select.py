"""The density query's two ways to list a slice's Gaussians (one block per
slice up to 16384 Gaussians, blocks of 256 Gaussians beyond) give the same
lists: a Gaussian that contributes nothing takes the call from one to the
other and changes no bit."""
import numpy as np
import pytest
import torch

import gemtest as gt
from paper_2509_25075_gb300 import synthetic as syn

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,max_B", [(32, 32), (48, 7)])
def test_both_forms(d, max_B):
    M = 16384
    th = syn.gaussians(syn.Workload("qs", d=d, M=M + 1, B=max_B, apix=1.2, s_lo=0.4, s_hi=2.0, seed=d))
    th[M, 10] = 0.0
    th[np.arange(0, M, 7), 2] *= 3.0  # some beyond the volume
    vol = []
    for n in (M, M + 1):
        w = syn.Workload("qs", d=d, M=n, B=max_B, apix=1.2, s_lo=0.4, s_hi=2.0, seed=d)
        ctx = gt.context(w)
        vol.append(ctx.gem_query(gt.to_dev(th[:n]), 1e-3))
        assert ctx.gem_status() == 0
        ctx.close()
    assert float(vol[0].max()) > 0
    assert torch.equal(vol[0], vol[1])


@pytest.mark.parametrize("tau_rel", [0.0, 1e-3])
@pytest.mark.parametrize("M,max_B", [(12500, 32), (12501, 32), (13312, 32), (13313, 32), (14335, 31), (16384, 25),
                                     (16385, 25), (16385, 32), (16639, 32), (16640, 32), (16641, 32)])
def test_forms_of_the_slices_agree(M, max_B, tau_rel):
    """A batch of slices takes every Gaussian in every slice up to 400000
    pairs, else lists of those that can matter, by one block per slice up to
    16384 Gaussians and by blocks of 256 beyond.  The volume is the same bits
    whatever the batch: max_B is compared with single slices, for counts on
    either side of the lines and of the forms' steps (1024, 256)."""
    d = 32
    w = syn.Workload("qf", d=d, M=M, B=max_B, apix=1.2, s_lo=0.4, s_hi=2.0, seed=M)
    th = syn.gaussians(w)
    z = np.array([-d / 2, d / 2 - 1, -d / 2 - 2.5, d / 2 + 1.5, -3 * d, 3 * d, 0.0]) * w.apix
    th[:, 2] = np.where(np.arange(M) % 2 == 0, z[np.arange(M) % 7], th[:, 2])
    th[3, 10] = -1.0  # contributes nothing
    P = gt.to_dev(th)
    vol = []
    for B in (1, max_B):
        ctx = gt.context(syn.Workload("qf", d=d, M=M, B=B, apix=1.2, seed=1), max_pairs=4 * M * B)
        vol.append(ctx.gem_query(P, tau_rel * w.tau_query / 1e-4))
        assert ctx.gem_status() == 0
        ctx.close()
    assert float(vol[0].max()) > 0
    assert torch.equal(vol[0], vol[1])
