"""A context is ready when gem_create returns, whatever is queued on the
default stream: its own stream may be a non-blocking one, which does not wait
for the default stream's clears of the context's counters."""
import pytest
import torch

import gemtest as gt
from paper_2509_25075_gb300 import binding
from paper_2509_25075_gb300 import synthetic as syn

pytestmark = pytest.mark.gpu

W = syn.Workload("create", d=32, M=900, B=3, apix=1.2, seed=61)


def test_context_is_ready_while_the_default_stream_is_busy():
    inp = gt.inputs(W)
    T = {k: gt.to_dev(v) for k, v in inp.items()}
    side = torch.cuda.Stream()
    out = []
    for busy in (False, True):
        torch.cuda.synchronize()
        if busy:
            torch.cuda._sleep(200_000_000)  # about 0.1 s
        ctx = binding.Context(W.d, W.apix, W.B, W.M, tau=W.tau, stream=side)
        # nothing of the context is left on the default stream
        assert torch.cuda.default_stream().query()
        with torch.cuda.stream(side):
            proj = torch.empty(W.B, W.d, W.d, device=gt.DEV)
            loss = torch.empty(1, dtype=torch.float64, device=gt.DEV)
            ctx.gem_project(T["params"], T["R"], T["t"], proj)
            ctx.gem_ctf_loss(proj, T["images"], ctf_params=T["ctf_params"], loss=loss)
            dist, idx = ctx.gem_nn_distance(T["params"], 2)
        side.synchronize()
        assert ctx.gem_status() == binding.GEM_OK
        out.append((proj, loss, dist, idx))
        ctx.close()
    for a, b in zip(*out):
        assert torch.equal(a, b)
