"""The density query's per-slice lists at the edges of its chunks (256
Gaussians) and batches, with Gaussians on, across and beyond the volume's
first and last slices, against the oracle."""
import numpy as np
import pytest

import gemtest as gt
import oracle
from paper_2509_25075_gb300 import synthetic as syn

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tau_rel", [0.0, 1e-3])
@pytest.mark.parametrize("M,max_B", [(1, 32), (255, 7), (256, 1), (257, 32), (700, 13)])
def test_slices_of_edge_gaussians(M, max_B, tau_rel):
    d, apix = 32, 1.2
    w = syn.Workload("qe", d=d, M=M, B=max_B, apix=apix, s_lo=0.4, s_hi=3.0, n_clusters=2, seed=M)
    th = syn.gaussians(w)
    z = np.array([-d / 2, d / 2 - 1, -d / 2 - 2.5, d / 2 + 1.5, -3 * d, 3 * d, 0.0]) * apix
    th[:, 2] = np.where(np.arange(M) % 2 == 0, z[np.arange(M) % 7], th[:, 2])
    if M > 10:
        th[3, 10] = -1.0  # contributes nothing
        th[5, 6:10] = 0.0
    full = oracle.query(th, d, apix, 0.0, 0)
    tau = tau_rel * float(full.max())
    ctx = gt.context(w)
    vol = ctx.gem_query(gt.to_dev(th), tau)
    assert ctx.gem_status() == 0
    ref = oracle.query(th, d, apix, tau, 0) if tau else full
    # a voxel may hold a few pairs that float32 puts on the other side of tau
    allow = 1e-5 * float(full.max()) + 3 * tau * (np.abs(vol.cpu().numpy() - ref) > 0.5 * tau) * (tau > 0)
    assert np.all(np.abs(vol.cpu().numpy() - ref) <= allow)
    assert np.sum(np.abs(vol.cpu().numpy() - ref) > 0.5 * tau) <= 3 if tau else True
    ctx.close()
