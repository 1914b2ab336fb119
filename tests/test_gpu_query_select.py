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
