"""The persistent chain kernel of fp32 heads at its edges (rows per group, ragged groups, columns per task, schedules longer
than a launch, feature tables that are no multiple of 16 bytes) against the float64 checker and the layer kernels."""
import numpy as np
import pytest

from paper_2411_11925_b200 import inputs as gen
from test_gpu_learned_variance import LvRound, _inputs as lv_inputs, _wl as lv_wl
from test_gpu_parity import _check, _wl

pytestmark = pytest.mark.gpu

CASES = [
    dict(B=1, gamma=1, T=2, draft=gen.HeadSpec(1, 128, 32), target=gen.HeadSpec(1, 128, 64)),                      # one row, 16 columns per CTA
    dict(B=5, gamma=8, T=3, draft=gen.HeadSpec(1, 256, 64), target=gen.HeadSpec(2, 384, 96)),                      # groups of 8 side by side, of 4 alone
    dict(B=7, gamma=3, T=3, cfg=True, cfg_scale=2.0, draft=gen.HeadSpec(2, 128, 64), target=gen.HeadSpec(1, 640, 96)),   # guided, last group ragged
    dict(B=19, gamma=11, T=2, cfg=True, cfg_scale=3.0, draft=gen.HeadSpec(1, 256, 64), target=gen.HeadSpec(1, 384, 64)),  # many groups of 16, ragged
    dict(B=3, gamma=2, T=2, cfg=True, cfg_scale=1.5, draft=gen.HeadSpec(1, 1024, 64), target=gen.HeadSpec(1, 1536, 64)),  # widest rows
    dict(B=2, gamma=2, T=3, draft=gen.HeadSpec(1, 128, 32, F=10), target=gen.HeadSpec(1, 256, 32, F=10)),          # features: 10 floats per row
]


@pytest.mark.parametrize("kw", CASES)
def test_f32_chain_matches_checker_and_fused_round_matches_the_calls(kw):
    from paper_2411_11925_b200.runner import DeviceRound
    inp = gen.make_round_inputs(_wl(**kw))
    _, a, _ = _check(inp, f"f32 chain {kw}")
    dr = DeviceRound(inp)
    dr.fused_round()
    b = dr.results()
    for k in ("x0", "mu1_q", "mu1_p", "logratio"):
        np.testing.assert_array_equal(a[k], b[k], err_msg=k)
    dr.ctx.close()


@pytest.mark.parametrize("T", [128, 129, 257])
def test_f32_schedules_longer_than_a_launch(T):
    # 128 steps per launch; the layer kernels are the reference (the same fp32 function summed in another order: a step's
    # rounding is about 1e-6 of a state of order one, and these ladders do not amplify it)
    from paper_2411_11925_b200 import api
    from paper_2411_11925_b200.runner import DeviceRound
    dr = DeviceRound(gen.make_round_inputs(_wl(B=3, gamma=2, T=T, cfg=True, cfg_scale=2.0, draft=gen.HeadSpec(1, 128, 32),
                                               target=gen.HeadSpec(1, 256, 32))))
    l0 = dr.ctx.launch_count()
    dr.draft_traj()
    assert dr.ctx.launch_count() - l0 == 2 + -(-T // 128)
    dr.ctx.sync()
    x, mu = dr.traj_x.clone(), dr.traj_mu.clone()
    dr.ctx.set_chain_mode(api.Context.CHAIN_LAYERS_PLAIN)
    dr.draft_traj()
    dr.ctx.sync()
    scale = float(dr.traj_x.abs().max())
    assert float((x - dr.traj_x).abs().max()) <= 2e-5 * scale and float((mu - dr.traj_mu).abs().max()) <= 2e-5 * scale
    dr.ctx.close()


@pytest.mark.parametrize("kw", [dict(B=1, gamma=1, T=1, cfg=False, cfg_scale=1.0), dict(B=9, gamma=5, T=6), dict(B=2, gamma=3, T=130)])
def test_f32_predicted_variances_match_the_layer_kernels(kw):
    from paper_2411_11925_b200 import api
    r = LvRound(lv_inputs(lv_wl(**kw)))
    got = []
    for mode in (api.Context.CHAIN_LAYERS, api.Context.CHAIN_LAYERS_PLAIN):
        r.ctx.set_chain_mode(mode)
        r.fused()
        got.append(r.results())
    for k in ("x0", "mu1_q", "lv1_q", "mu1_p", "lv1_p"):
        assert float(np.max(np.abs(got[0][k] - got[1][k]))) <= 2e-5 * max(1.0, float(np.abs(got[1][k]).max())), k
    # half_logdet: T C / 2 variance terms of order 10
    for k in ("hld_q", "hld_p"):
        assert float(np.max(np.abs(got[0][k] - got[1][k]))) <= 1e-6 * max(1.0, float(np.abs(got[1][k]).max())) * kw["T"] ** 0.5 + 1e-4, k
    r.ctx.close()


@pytest.mark.parametrize("W,R,cfg", [(896, 91 * 32, False), (1536, 53 * 16, True), (2048, 512, False)])
def test_most_rows_of_the_chain_kernel_and_one_more(W, R, cfg):
    # 637, 636 and 256 tiles (groups of 16, 8 and 4 head rows); one token more runs as layer kernels, the same fp32 function summed in another order
    from paper_2411_11925_b200 import api
    from paper_2411_11925_b200.runner import DeviceRound
    for rows, chain in ((R, True), (R + 1, False)):
        dr = DeviceRound(gen.make_round_inputs(_wl(B=rows, gamma=1, T=2, cfg=cfg, cfg_scale=2.0, draft=gen.HeadSpec(1, W, 32), target=gen.HeadSpec(1, 128, 32))))
        l0 = dr.ctx.launch_count()
        dr.draft()
        assert (dr.ctx.launch_count() - l0 == 3) == chain, (rows, dr.ctx.launch_count() - l0)
        dr.ctx.sync()
        x0 = dr.x0.clone()
        dr.ctx.set_chain_mode(api.Context.CHAIN_LAYERS_PLAIN)
        dr.draft()
        dr.ctx.sync()
        assert float((x0 - dr.x0).abs().max()) <= 2e-5 * float(dr.x0.abs().max())
        dr.ctx.close()
