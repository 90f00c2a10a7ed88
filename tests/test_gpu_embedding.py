"""The timestep embedding's sums run in ascending order of k: part of the results of every 16-bit chain (an ulp of the embedding
flips roundings of the condition vector) and of the plain fp32 layer kernels."""
import numpy as np
import pytest
import torch

from paper_2411_11925_b200 import inputs as gen
from test_gpu_parity import _check, _wl

pytestmark = pytest.mark.gpu


def _cancelling(rng, rows, K):
    """Rows with 2^25 at k0, 1 at k1, -2^25 at k2, k0 < k1 < k2: times equal positive factors below one, ascending order sums to
    exactly zero (the middle term is below half an ulp of the first), any order that meets the outer two first does not."""
    w = np.zeros((rows, K), np.float32)
    for n in range(rows):
        k0, k1, k2 = np.sort(rng.choice(K, 3, replace=False))
        w[n, k0], w[n, k1], w[n, k2] = 2.0 ** 25, 1.0, -2.0 ** 25
    return w


@pytest.mark.parametrize("op,mode,L,W,R,T,F", [
    ("f16", 0, 2, 512, 5, 3, 256),         # group chain kernel
    ("f16", 0, 1, 1024, 300, 2, 10),       # layer kernels; feature rows of 40 bytes
    ("f16", 0, 2, 1024, 300, 2, 10),       # wide chain kernel
    ("bf16", 2, 1, 256, 3, 65, 30),        # layer kernels; more steps than two tiles of rows
    ("f16", 2, 1, 128, 3, 64, 256),
    ("f32", 2, 1, 384, 3, 9, 33),
])
def test_sums_run_in_ascending_order(op, mode, L, W, R, T, F):
    from paper_2411_11925_b200 import api
    rng = np.random.default_rng(W + T)
    w = gen.make_head_weights(gen.HeadSpec(L, W, 64, F=F), rng, op != "f32")
    w["bt1"] = np.full(W, 0.5, np.float32)           # hidden layer: SiLU(0.5) everywhere
    zero = {**w, "Wt1": np.zeros((W, F), np.float32), "Wt2": np.zeros((W, W), np.float32)}
    hard = {**w, "Wt1": _cancelling(rng, W, F), "Wt2": _cancelling(rng, W, W)}
    dev = torch.device("cuda", 0)
    ctx = api.Context(0)
    ctx.set_chain_mode(mode)
    co = api.ddpm_coefficients(gen.beta_linear(T))
    sched = api.Schedule(co["a"], co["b"], co["sigma"], torch.full((T, F), 0.75, device=dev))
    z, x_T, eps = (torch.randn(s, device=dev, generator=torch.Generator(dev).manual_seed(1)) for s in ((R, 64), (R, 16), (T, R, 16)))
    got = []
    for weights in (zero, hard):
        x0, mu1 = torch.zeros(R, 16, device=dev), torch.zeros(R, 16, device=dev)
        ctx.csd_draft_denoise(api.Head(ctx, weights, op), sched, R, False, 1.0, z, x_T, eps, x0, mu1)
        ctx.sync()
        got.append((x0, mu1))
    assert float(got[0][0].abs().max()) > 0.0
    assert bool((got[0][0] == got[1][0]).all()) and bool((got[0][1] == got[1][1]).all())
    ctx.close()


@pytest.mark.parametrize("T,F", [(1, 256), (8, 10), (9, 256), (63, 250), (65, 34)])
def test_embedding_edges_match_checker(T, F):
    # a tile has 8 rows below 64 steps, 32 from there on; F no multiple of 32, of 4
    kw = dict(B=3, gamma=2, T=T, bf16=True, draft=gen.HeadSpec(1, 128, 64, F=F), target=gen.HeadSpec(1, 384, 64, F=F))
    _check(gen.make_round_inputs(_wl(**kw)), f"embedding {T} {F}")
