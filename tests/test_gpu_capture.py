"""Calls captured into CUDA graphs: a graph carries everything that it needs from the host, and graphs of one context may run side
by side as far as they share no workspace."""
import numpy as np
import pytest
import torch

from paper_2411_11925_b200 import inputs as gen
from test_gpu_parity import _wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kw", [
    dict(B=3, gamma=2, T=40, bf16=True, cfg=True, cfg_scale=2.0, draft=gen.HeadSpec(1, 512, 64), target=gen.HeadSpec(1, 512, 64)),   # group chain
    dict(B=3, gamma=2, T=5, draft=gen.HeadSpec(1, 128, 64), target=gen.HeadSpec(1, 128, 64)),                                     # fp32 chain
])
def test_captured_draft_call_replays_after_its_host_arrays_are_gone(kw):
    from paper_2411_11925_b200 import api
    from paper_2411_11925_b200.runner import DeviceRound
    inp = gen.make_round_inputs(_wl(**kw))
    side = torch.cuda.Stream()
    dr = DeviceRound(inp, ctx=api.Context(0, side))
    torch.cuda.synchronize()
    dr.draft()                                        # workspaces
    dr.ctx.sync()
    want = dr.x0.clone()
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=side):
        dr.draft()
    for k in ("a", "b", "sigma"):
        getattr(dr.sched_q, k)[:] = np.nan            # the caller's coefficients: copied before the call returns
    junk = [np.full(3 * kw["T"] + i % 8, np.nan, np.float32) for i in range(2000)]      # (and whatever the call had on the heap)
    dr.x0.zero_()
    torch.cuda.synchronize()
    g.replay()
    torch.cuda.synchronize()
    assert len(junk) == 2000 and bool((dr.x0 == want).all())
    dr.ctx.close()
