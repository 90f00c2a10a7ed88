"""Calls of few rows where the device has little memory left: the group chain kernel's chunks get shorter, with the same bits, and
where none fits the layer kernels run."""
import pytest
import torch

from paper_2411_11925_b200 import inputs as gen
from _parity import TOL_X
from test_gpu_parity import _wl

pytestmark = pytest.mark.gpu


def test_few_rows_with_little_memory_left():
    from paper_2411_11925_b200 import api
    from paper_2411_11925_b200.runner import DeviceRound
    # 64 tokens with guidance, two 1024-wide blocks, 60 steps: 16 MB of condition vectors, 2 x 252 MB of condition products; one step 2 x 8 MB
    wl = _wl(bf16=True, B=64, gamma=1, T=60, cfg=True, cfg_scale=2.0, draft=gen.HeadSpec(2, 1024, 64), target=gen.HeadSpec(1, 128, 64))
    inp = gen.make_round_inputs(wl)
    ref = DeviceRound(inp)
    launches = []
    for mode in (api.Context.CHAIN_LAYERS_PLAIN, api.Context.CHAIN_LAYERS):     # (both ways' kernels are loaded before memory is taken)
        ref.ctx.set_chain_mode(mode)
        l0 = ref.ctx.launch_count()
        ref.draft()
        ref.ctx.sync()
        launches.append(ref.ctx.launch_count() - l0)
    want = ref.x0.clone()
    tight, none = DeviceRound(inp), DeviceRound(inp)
    got = torch.empty_like(want)
    torch.cuda.synchronize()
    hog = []

    def leave(mb):
        while (free := torch.cuda.mem_get_info()[0]) > (mb + 4) << 20:
            hog.append(torch.empty((free - (mb << 20)) >> 21 << 21, dtype=torch.uint8, device="cuda"))

    try:
        leave(160)
        l0 = tight.ctx.launch_count()
        tight.draft()
        tight.ctx.sync()
        n = tight.ctx.launch_count() - l0
        assert launches[1] < n < launches[1] + 40, (launches, n)                # the same kernels, more chunks
        got.copy_(tight.x0)
        assert bool((got == want).all())
        tight.ctx.close()
        leave(24)                                                               # room for workspace and condition vectors, not for products
        l0 = none.ctx.launch_count()
        none.draft()
        none.ctx.sync()
        assert none.ctx.launch_count() - l0 == launches[0]
        assert float((none.x0 - want).abs().max()) <= TOL_X["f16"] / 4
    finally:
        hog.clear()
        torch.cuda.empty_cache()
    for d in (ref, none):
        d.ctx.close()
