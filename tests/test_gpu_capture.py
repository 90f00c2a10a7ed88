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


def test_resampling_graphs_of_one_context_side_by_side():
    from paper_2411_11925_b200 import api
    B, gamma, C, cap = 2048, 1, 16, 2
    side = torch.cuda.Stream()
    ctx = api.Context(0, side)
    rng = torch.Generator("cuda").manual_seed(3)
    N = lambda *s: torch.randn(s, device="cuda", generator=rng)
    calls = []
    for i in range(3):
        mu_p = N(B * gamma, C)
        mu_q = mu_p + 0.002 * (i + 1) * N(B * gamma, C)
        out = dict(x=torch.zeros(B, C, device="cuda"), hits=torch.zeros(1, dtype=torch.int32, device="cuda"),
                   **{k: torch.zeros(B, dtype=torch.int32, device="cuda") for k in ("n", "flags")})
        args = (torch.zeros(B, dtype=torch.int32, device="cuda"), mu_p, mu_q, N(B, cap, C), torch.rand(B, cap, device="cuda", generator=rng).clamp(1e-6, 1 - 1e-6))
        calls.append((lambda a=args, o=out: ctx.csd_resample(B, gamma, C, cap, 0.0, 0.01, 0.01, *a, o["x"], o["n"], o["flags"], o["hits"]), out))
    torch.cuda.synchronize()
    want = []
    for call, out in calls:
        call()
        ctx.sync()
        want.append(int(((out["flags"] & 2) != 0).sum()))
        assert int(out["hits"].item()) == want[-1] > 0
    torch.cuda.synchronize()
    graphs = []
    for call, _ in calls[:2]:
        graphs.append(torch.cuda.CUDAGraph())
        with torch.cuda.graph(graphs[-1], stream=side):
            call()
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    torch.cuda.synchronize()
    for _ in range(50):
        for g, s in zip(graphs, streams):
            with torch.cuda.stream(s):
                g.replay()
        calls[2][0]()                                 # and the context's own stream
    torch.cuda.synchronize()
    assert [int(o["hits"].item()) for _, o in calls] == want
    calls[2][0]()
    ctx.sync()
    assert int(calls[2][1]["hits"].item()) == want[2]
    ctx.close()
