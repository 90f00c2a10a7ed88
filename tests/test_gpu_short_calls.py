"""Edges of the short calls' kernels: proposals per pass, components per lane group, mixtures too large for shared memory,
unaligned rows, one block or several."""
import numpy as np
import pytest
import torch

from oracle import csd_oracle as orc
from test_gpu_gmm import test_gmm_round_matches_checker as check_gmm_round

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,gamma,Kq,Kp,C,cap,close", [
    (1, 1, 1, 1, 1, 1, 0.1),            # smallest of everything
    (3, 2, 16, 17, 17, 65, 0.0),        # one component more than a half-warp, 32-wide coordinates, one proposal in a second pass
    (5, 3, 17, 17, 16, 64, 0.02),       # exactly one pass of proposals
    (4, 5, 33, 2, 3, 200, 0.0),         # more components than a warp on one side
    (2, 2, 100, 100, 32, 70, 0.02)])    # shared tables would need 64 KB: formed on the fly
def test_gmm_kernel_edges_match_checker(B, gamma, Kq, Kp, C, cap, close):
    check_gmm_round(B, gamma, Kq, Kp, C, cap, close)


@pytest.mark.parametrize("B,C,cap,offset", [(1, 1, 1, 0), (4, 16, 32, 0), (5, 16, 33, 1), (7, 3, 64, 0), (33, 15, 200, 0)])
def test_resample_edges_match_checker(B, C, cap, offset):
    from paper_2411_11925_b200 import api
    dev = torch.device("cuda", 0)
    ctx = api.Context(0)
    rng = np.random.default_rng(100 * B + cap)
    gamma = 3
    mu_p = rng.standard_normal((B * gamma, C)).astype(np.float32)
    mu_q = (mu_p + 0.004 * rng.standard_normal(mu_p.shape)).astype(np.float32)
    n_acc = rng.integers(0, gamma + 1, B).astype(np.int32)
    n_acc[0] = 1
    xi = rng.standard_normal((B, cap, C)).astype(np.float32)
    v = rng.random((B, cap)).astype(np.float32).clip(1e-7, 1 - 1e-7)
    ref = orc.resample(n_acc, mu_p.astype(np.float64), mu_q.astype(np.float64), 0.01, 0.0102, -0.1, xi, v, gamma, cap)
    t = lambda a: torch.from_numpy(a).to(dev)
    d_xi = torch.zeros(xi.size + offset, device=dev)[offset:].view(xi.shape)     # offset 1: rows not on 16-byte boundaries
    d_xi.copy_(t(xi))
    x_new = torch.full((B, C), 7.0, device=dev)
    n_prop, flags = (torch.zeros(B, dtype=torch.int32, device=dev) for _ in range(2))
    hits = torch.full((1,), 99, dtype=torch.int32, device=dev)
    for _ in range(2):                                                           # the tally starts from zero again
        ctx.csd_resample(B, gamma, C, cap, -0.1, 0.01, 0.0102, t(n_acc), t(mu_p), t(mu_q), d_xi, t(v), x_new, n_prop, flags, hits)
    ctx.sync()
    g_prop, g_flags, g_x = n_prop.cpu().numpy(), flags.cpu().numpy(), x_new.cpu().numpy()
    same = g_prop == ref["n_prop"]
    assert same.mean() >= 0.96, (g_prop, ref["n_prop"])      # a threshold within rounding of v may flip a proposal (33 sequences: one)
    np.testing.assert_array_equal(g_flags[same], ref["flags"][same])
    res = same & (n_acc < gamma)
    np.testing.assert_allclose(g_x[res], ref["x_new"][res], atol=1e-6)           # |x'| <= 6: a few fp32 ulp
    assert np.all(g_x[n_acc == gamma] == 7.0) and np.all(g_prop[n_acc == gamma] == 0)
    assert int(hits.item()) == int(((g_flags & 2) != 0).sum())
    ctx.close()
