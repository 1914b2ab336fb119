"""Depth order at the sizes where the sort changes form (one CTA per row up to
8192 keys, or 24576 with 32 rows and more) and at ragged ends of its
stretches: every tile's list holds the same Gaussians as without the sort, in
ascending depth within the key's step."""
import numpy as np
import pytest
import torch

import gemtest as gt
from paper_2509_25075_gb300 import synthetic as syn

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,B", [(1, 1), (31, 2), (33, 1), (1023, 1), (1025, 2), (4097, 1), (8192, 1), (8193, 1),
                                 (20001, 32), (24576, 32), (24577, 32)])
def test_depth_order(M, B):
    w = syn.Workload("ds", d=32, M=M, B=B, apix=1.2, seed=M % 97)
    inp = gt.inputs(w)
    R, t, P = (gt.to_dev(inp[k]) for k in ("R", "t", "params"))
    z = torch.einsum("bk,mk->bm", R[:, 2].double(), P[:, :3].double())
    step = 2.0 * w.d * w.apix / 65536
    got = {}
    for zsort in (1, 0):
        ctx = gt.context(w, zsort=zsort)
        proj = torch.empty(B, w.d, w.d, device=gt.DEV)
        ctx.gem_project(P, R, t, proj)
        assert ctx.gem_status() == 0
        ts, lst = ctx.gem_inspect_bins()
        tile = torch.repeat_interleave(torch.arange(len(ts) - 1, device=gt.DEV), ts[1:] - ts[:-1])
        got[zsort] = (ts, tile, lst.long())
        ctx.close()
    assert torch.equal(got[1][0], got[0][0])
    key = [torch.sort(tile * M + lst).values for _, tile, lst in (got[1], got[0])]
    assert torch.equal(key[0], key[1])
    ts, tile, lst = got[1]
    depth = z[tile // 4, lst]
    same = tile[1:] == tile[:-1]
    assert (depth[1:] - depth[:-1] >= -step - 1e-4)[same].all()
