"""Performance cases of the continuous-speculative-decoding library.

Each case is work a decoding program has the library do, through the calls of `paper_2411_11925_b200.api`: whole
speculative rounds, the draft calls of an autoregressive loop, the single-path criterion, the accept / resample calls
and the Gaussian-mixture heads.  Sizes are those of the workload table in `paper_2411_11925_b200.inputs` and of the
tests, or generic odd ones.  A model (context and heads) lives as long as the process, as in a serving program; what
changes from request to request - condition vectors, noise, uniforms - is made from the seed.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2411_11925_b200 import api, inputs as gen

C_TOKEN = 16          # latent token dimension of every head below
GUIDANCE = 3.0        # guidance scale of the workload table
CAP = 64              # proposals of the resampling loop

# Head pairs (draft, target): blocks, width, condition dimension.  "stress" perturbs the target's weights.
PAIRS = {
    "tiny": ((1, 128, 256), (2, 256, 256)),
    "odd": ((1, 256, 128), (2, 384, 192)),
    "mar": ((3, 1024, 768), (6, 1024, 1024)),
    "large": ((6, 1024, 1024), (12, 1536, 1280)),
    "stress": ((8, 1024, 1024), (8, 1024, 1024)),
}
STRESS_STD = 0.05
MODES = {"default": api.Context.CHAIN_LAYERS, "small_batch": api.Context.CHAIN_SMALL_BATCH}


def _case(name, call, B, gamma, *, pair="", T=0, guided=True, operand="f16", mode="default", C=C_TOKEN, K=0):
    c = {"call": call, "B": B, "gamma": gamma, "C": C}
    if pair:
        c.update(pair=pair, T=T, guided=guided, operand=operand, mode=mode)
    if K:
        c["K"] = K
    return {"name": name, **c} if name else c


def listed():
    return [
        # the ratio / accept / resample calls on their own, for a program that holds the final-step means already
        _case("accept_resample", "accept_resample", 64, 8),
        # a round of explicit mixture heads (no diffusion chain): sample, verify, resample; odd batch
        _case("gmm_round", "gmm_round", 37, 7, K=6),
        # the smallest round of the workload table: fp32 heads, one sequence
        _case("round_tiny_f32", "round", 1, 4, pair="tiny", T=10, guided=False, operand="f32"),
        # the autoregressive draft loop: one position of 64 sequences per call, in the mode meant for it
        _case("draft_position", "draft", 64, 1, pair="mar", T=100, mode="small_batch"),
        # one position of a few sequences, library defaults, no guidance, bf16 operands
        _case("draft_position_few", "draft", 11, 1, pair="mar", T=50, guided=False, operand="bf16"),
        # the headline round (256 x 256 images)
        _case("round_mar256", "round", 64, 8, pair="mar", T=100),
        # the same round from and to host buffers, as a program without device tensors calls it
        _case("round_host", "round_host", 64, 8, pair="mar", T=100),
        # a ragged batch with the bonus position riding along
        _case("round_bonus_odd", "round_bonus", 37, 7, pair="mar", T=100),
        # heads that predict their variances
        _case("round_lv", "round_lv", 48, 8, pair="mar", T=100),
        # the exact single-path criterion on the draft's recorded trajectory
        _case("single_path", "single_path", 64, 8, pair="mar", T=100),
        # no guidance, long batch, draft = perturbed target, bf16 operands
        _case("round_ar_stress", "round", 256, 16, pair="stress", T=50, guided=False, operand="bf16"),
        # the largest round of the workload table
        _case("round_large_target", "round", 128, 16, pair="large", T=100),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    most = work(listed()[-1])["flops"]
    while True:
        kind = rng.choice(["accept_resample", "gmm_round", "f32", "draft", "draft", "round", "round", "round_host", "round_bonus",
                           "round_lv", "single_path"])
        gamma = _log_int(rng, 1, 32)
        if kind == "accept_resample":
            return _case("", kind, _log_int(rng, 1, 4096), gamma, C=rng.randint(3, 16))
        if kind == "gmm_round":
            return _case("", kind, _log_int(rng, 1, 1024), gamma, C=rng.randint(2, 32), K=_log_int(rng, 1, 24))
        T = _log_int(rng, 10, 100)
        guided = rng.random() < 0.7
        if kind == "f32":
            c = _case("", "round", _log_int(rng, 1, 48), _log_int(rng, 1, 16), pair=rng.choice(["tiny", "odd"]), T=T, guided=guided,
                      operand="f32")
        elif kind == "draft":
            mode = rng.choice(["default", "small_batch"])
            c = _case("", kind, _log_int(rng, 1, 64), 1, pair=rng.choice(["mar", "large", "stress"]), T=T, guided=guided,
                      operand=rng.choice(["f16", "f16", "bf16"]), mode=mode)
        else:
            c = _case("", kind, _log_int(rng, 4, 256), gamma, pair=rng.choice(["mar", "mar", "large", "stress"]), T=T, guided=guided,
                      operand=rng.choice(["f16", "f16", "bf16"]))
        if work(c)["flops"] <= most:
            return c


# ------------------------------------------------------------------------------------------------ work and tolerance
def _head_params(spec, out_cols):
    L, W, Dz = spec
    F = 256
    return W * Dz + W * F + W * W + 5 * L * W * W + 2 * W * W + (C_TOKEN + out_cols) * W + (5 * L + 8) * W


def _row_step_flops(spec, out_cols):
    L, W, _ = spec
    return 2.0 * W * (C_TOKEN + out_cols + (5 * L + 2) * W)


def work(case):
    B, g, C = case["B"], case["gamma"], case["C"]
    R = B * g
    if case["call"] == "accept_resample":
        # x0, two means and u in, log-ratios and counts out; one proposal per sequence
        n = 3 * R * C + R + B * (C + 1) + R + 4 * B + B * C
        return {"bytes": 4.0 * n, "flops": 6.0 * R * C + 8.0 * B * C}
    if case["call"] == "gmm_round":
        K = case["K"]
        n = 2 * R * K * (2 * C + 1) + R * (2 + C) + B * (C + 2) + 2 * R + R * C + 4 * B + B * C
        return {"bytes": 4.0 * n, "flops": 2.0 * R * K * 6 * C + 2.0 * B * K * 6 * C}
    T, rep = case["T"], 2 if case["guided"] else 1
    q, p = PAIRS[case["pair"]]
    wsize = 4.0 if case["operand"] == "f32" else 2.0
    out_cols = 2 * C if case["call"] == "round_lv" else C
    Rp = R + B if case["call"] == "round_bonus" else R
    nbytes = wsize * _head_params(q, out_cols) + 4.0 * (R * rep * q[2] + R * C + T * R * C + 2 * R * C)
    flops = float(rep) * R * T * _row_step_flops(q, out_cols)
    if case["call"] == "single_path":
        nbytes += 4.0 * (2 * T + 1) * R * C
    if case["call"] != "draft":
        nbytes += wsize * _head_params(p, out_cols) + 4.0 * (Rp * rep * p[2] + (Rp - R) * (T + 1) * C + 2 * R * C + 2 * R + B * (2 * C + 6))
        flops += float(rep) * Rp * T * _row_step_flops(p, out_cols)
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    operand = case.get("operand", "f32")
    if operand == "f32":
        # fp32 sums throughout; a decision may flip on a tie
        return {"rel": 2e-5, "max": 1e-3, "differ": 0.005}
    # 16-bit operands whose rounding a chain of T dependent steps carries on
    if operand == "f16":
        return {"rel": 5e-3, "max": 0.2, "differ": 0.01}
    return {"rel": 3e-2, "max": 0.8, "differ": 0.01}


# ------------------------------------------------------------------------------------------------ the long-lived part
_CONTEXTS, _HEADS, _WEIGHTS = {}, {}, {}


def _context(mode):
    if mode not in _CONTEXTS:
        _CONTEXTS[mode] = api.Context(0)
        _CONTEXTS[mode].set_chain_mode(MODES[mode])
    return _CONTEXTS[mode]


def _weights(pair, side, bf16, var_out):
    """Random-init weights by the recipe of the workload table: the same for every seed."""
    key = (pair, side, bf16, var_out)
    if key not in _WEIGHTS:
        _WEIGHTS.clear()      # one set of host weights at a time
        L, W, Dz = PAIRS[pair][side]
        rng = np.random.Generator(np.random.PCG64(1000 * sorted(PAIRS).index(pair) + side))
        if pair == "stress" and side == 0:
            base = _weights(pair, 1, bf16, var_out)
            w = gen.perturb_head_weights(base, rng, STRESS_STD, bf16)
        else:
            w = gen.make_head_weights(gen.HeadSpec(L, W, Dz, C=C_TOKEN, var_out=var_out), rng, bf16)
        _WEIGHTS[key] = w
    return _WEIGHTS[key]


def _head(mode, pair, side, operand, var_out):
    key = (mode, pair, side, operand, var_out)
    if key not in _HEADS:
        _HEADS[key] = api.Head(_context(mode), _weights(pair, side, operand != "f32", var_out), operand, var_out)
    return _HEADS[key]


# ------------------------------------------------------------------------------------------------ one request's state
def _uniform(shape, g):
    return torch.rand(shape, generator=g, device="cuda").clamp_(2.0 ** -24, 1.0 - 2.0 ** -24)


def _zeros(*shape, dtype=torch.float32):
    return torch.zeros(*shape, dtype=dtype, device="cuda")


def _scan_outputs(s, B, gamma, C):
    s.update(logratio=_zeros(B, gamma), n_accept=_zeros(B, dtype=torch.int32), accept_mask=_zeros(B, dtype=torch.int32),
             x_new=_zeros(B, C), n_prop=_zeros(B, dtype=torch.int32), flags=_zeros(B, dtype=torch.int32),
             cap_hits=_zeros(1, dtype=torch.int32))


SCAN_OUT = ("logratio", "n_accept", "accept_mask", "x_new", "n_prop", "flags", "cap_hits")


def prepare(case, seed):
    B, gamma, C = case["B"], case["gamma"], case["C"]
    R = B * gamma
    g = torch.Generator(device="cuda").manual_seed(seed)
    normal = lambda *shape: torch.randn(shape, generator=g, device="cuda")
    s = {"case": case, "call": case["call"], "B": B, "gamma": gamma, "C": C, "R": R}
    s["u"], s["xi"], s["v"] = _uniform((B, gamma), g), normal(B, CAP, C), _uniform((B, CAP), g)
    if case["call"] == "accept_resample":
        # draft and target means a fraction of sigma_1 apart, as with a good draft: some drafts accepted, some not
        s["ctx"], s["sigma"] = _context("default"), 0.01
        s["mu1_q"] = normal(R, C)
        s["mu1_p"] = s["mu1_q"] + 0.4 * s["sigma"] * normal(R, C)
        s["x0"] = s["mu1_q"] + s["sigma"] * normal(R, C)
        _scan_outputs(s, B, gamma, C)
        return s
    if case["call"] == "gmm_round":
        K = case["K"]
        s["ctx"] = _context("default")
        s["q"] = (normal(R, K), 2.0 * normal(R, K, C), 0.3 * normal(R, K, C) - 0.5)
        s["p"] = tuple((a + d * normal(*a.shape)).contiguous() for a, d in zip(s["q"], (0.3, 0.2, 0.05)))
        s["u_comp"], s["noise"], s["w"] = _uniform((R,), g), normal(R, C), _uniform((B, CAP), g)
        s["x"], s["comp"] = _zeros(R, C), _zeros(R, dtype=torch.int32)
        _scan_outputs(s, B, gamma, C)
        return s
    T, guided, operand, mode, lv = case["T"], case["guided"], case["operand"], case["mode"], case["call"] == "round_lv"
    rep = 2 if guided else 1
    s["ctx"], s["guided"], s["scale"], s["T"] = _context(mode), guided, GUIDANCE if guided else 1.0, T
    tfeat = torch.from_numpy(gen.timestep_features(T, 256)).cuda()
    if lv:
        co = api.lv_ddpm_coefficients(gen.beta_linear(T))
        s["sched"] = api.ScheduleLV(co["a"], co["b"], co["lv_min"], co["lv_max"], tfeat)
    else:
        co = api.ddpm_coefficients(gen.beta_linear(T))
        s["sched"] = api.Schedule(co["a"], co["b"], co["sigma"], tfeat)

    def condition(rows, side):
        z = normal(rows * rep, PAIRS[case["pair"]][side][2])
        return z if operand == "f32" else z.bfloat16().float()

    sides = (0,) if case["call"] == "draft" else (0, 1)
    for side in sides[::-1]:
        s["head_" + "qp"[side]] = _head(mode, case["pair"], side, operand, lv)
    for side in sides:
        s["z_" + "qp"[side]] = condition(R, side)
    s["x_T"], s["eps"] = normal(R, C), normal(T, R, C)
    s["x0"], s["mu1_q"], s["mu1_p"] = (_zeros(R, C) for _ in range(3))
    _scan_outputs(s, B, gamma, C)
    if lv:
        s.update({n: _zeros(R, C) for n in ("lv1_q", "lv1_p")}, **{n: _zeros(R) for n in ("hld_q", "hld_p", "log_sigma_rows")})
    if case["call"] == "round_bonus":
        s["z_next"], s["x_T_next"], s["eps_next"] = condition(B, 1), normal(B, C), normal(T, B, C)
        s["x_bonus"], s["taken"] = _zeros(B, C), _zeros(B, dtype=torch.int32)
    if case["call"] == "single_path":
        s["traj_x"], s["traj_mu"] = _zeros(T + 1, R, C), _zeros(T, R, C)
    if case["call"] == "round_host":
        for n in ("z_q", "z_p", "x_T", "eps", "u", "xi", "v", "x0", "mu1_q", "mu1_p") + SCAN_OUT:
            s[n] = s[n].cpu().pin_memory()
    return s


def _get(s, *names):
    return {n: s[n] for n in names}


def run(s):
    ctx, call, B, gamma, C, R = s["ctx"], s["call"], s["B"], s["gamma"], s["C"], s["R"]
    scan = tuple(s[n] for n in SCAN_OUT)
    if call == "accept_resample":
        ctx.csd_accept_scan(B, gamma, C, 0.0, s["sigma"], s["sigma"], s["x0"], s["mu1_q"], s["mu1_p"], s["u"], *scan[:3])
        ctx.csd_resample(B, gamma, C, CAP, 0.0, s["sigma"], s["sigma"], s["n_accept"], s["mu1_p"], s["mu1_q"], s["xi"], s["v"],
                         *scan[3:])
        return _get(s, *SCAN_OUT)
    if call == "gmm_round":
        ctx.csd_gmm_draft_sample(R, C, s["q"], s["u_comp"], s["noise"], s["x"], s["comp"])
        ctx.csd_gmm_verify(B, gamma, C, s["q"], s["p"], s["x"], s["u"], *scan[:3])
        ctx.csd_gmm_resample(B, gamma, C, CAP, s["q"], s["p"], s["n_accept"], s["w"], s["xi"], s["v"], *scan[3:])
        return _get(s, "x", "comp", *SCAN_OUT)
    head, sched, common = (s["head_q"], s.get("head_p")), s["sched"], (s["guided"], s["scale"])
    if call == "draft":
        ctx.csd_draft_denoise(head[0], sched, R, *common, s["z_q"], s["x_T"], s["eps"], s["x0"], s["mu1_q"])
        return _get(s, "x0", "mu1_q")
    if call == "single_path":
        ctx.csd_draft_denoise_traj(head[0], sched, R, *common, s["z_q"], s["x_T"], s["eps"], s["traj_x"], s["traj_mu"])
        ctx.csd_verify_single_path(head[1], sched, sched, B, gamma, *common, s["z_p"], s["traj_x"], s["traj_mu"], s["u"], 0, *scan[:3])
        return _get(s, "traj_x", "traj_mu", *SCAN_OUT[:3])
    inputs = (*head, sched, sched, B, gamma, *common, CAP, s["z_q"], s["z_p"], s["x_T"], s["eps"], s["u"], s["xi"], s["v"])
    if call == "round_lv":
        ctx.csd_round_lv(*inputs, s["x0"], s["mu1_q"], s["lv1_q"], s["hld_q"], s["mu1_p"], s["lv1_p"], s["hld_p"],
                         s["log_sigma_rows"], *scan)
        return _get(s, "x0", "mu1_q", "lv1_q", "hld_q", "mu1_p", "lv1_p", "hld_p", "log_sigma_rows", *SCAN_OUT)
    means = (s["x0"], s["mu1_q"], s["mu1_p"])
    if call == "round_bonus":
        ctx.csd_round_bonus(*inputs, s["z_next"], s["x_T_next"], s["eps_next"], *means, *scan, s["x_bonus"], s["taken"])
        return _get(s, "x0", "mu1_q", "mu1_p", *SCAN_OUT, "x_bonus", "taken")
    (ctx.csd_round_host if call == "round_host" else ctx.csd_round)(*inputs, *means, *scan)
    return _get(s, "x0", "mu1_q", "mu1_p", *SCAN_OUT)
