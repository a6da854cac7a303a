"""Timed workloads of the HeatKV hot path: what programs built on this library have it do.

Two kinds of work.  `generate`: one batch of images through the attention + cache path of a stack of layers, from
opening the sequences to closing them, every scale and layer in generation order (`Session.generate`).  `calibrate`:
the attention mass per source scale (Eq. 2) of one batch of samples, layer by layer, in the form the caller needs: from
recorded activations in one call per layer ("recorded"), inside a running model that needs the attention output too
("forward"), step by step without an output ("steps"), or where nothing may be allocated ("static").

The calibrated scores and with them the eviction schedule belong to the model, so they depend on the case alone; the
activations come from the seed.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2605_14877_b200 as hk
from paper_2605_14877_b200.sweep import Session

SIDES_13 = (1, 2, 4, 6, 8, 12, 16, 20, 24, 32, 40, 48, 64)        # a 1024 x 1024 image
SERVING_BUDGETS = (1 / 5, 1 / 10, 1 / 20, 1 / 40)
SINKS = 3
MAX_FLOPS = 8.2e12                                                # the largest listed case


def _grid(sides, aspect=1.0):
    """Scale list as text, "WxH,WxH,..": square sides, or the same areas at another aspect ratio."""
    wh = [(max(1, round(s * math.sqrt(aspect))), max(1, round(s / math.sqrt(aspect)))) for s in sides]
    return ",".join("%dx%d" % p for p in wh)


def _tokens(case):
    return [int(p.split("x")[0]) * int(p.split("x")[1]) for p in case["scales"].split(",")]


def _generate(name, scales, L, H, n_seq, budget, d=128, cache="bf16", layout="paged", fused=True, bias=False,
              token_major=False, sinks=SINKS):
    return {"name": name, "kind": "generate", "scales": scales, "L": L, "H": H, "d": d, "n_seq": n_seq, "sinks": sinks,
            "budget": budget, "cache": cache, "layout": layout, "fused": fused, "bias": bias, "token_major": token_major}


def _calibrate(name, scales, L, H, n_seq, calls, d=128, bias=False, token_major=False):
    return {"name": name, "kind": "calibrate", "scales": scales, "L": L, "H": H, "d": d, "n_seq": n_seq, "sinks": SINKS,
            "calls": calls, "bias": bias, "token_major": token_major}


def listed():
    full = _grid(SIDES_13)
    return [
        # One small image through one small layer: four launches, nothing but latency.  Budget -1: per-head fractions.
        _generate("tiny_image", _grid((1, 2, 4, 8)), L=1, H=4, d=64, n_seq=1, budget=-1.0, sinks=0),
        # A 256 x 256 preview of one prompt (conditional and unconditional sequence): only small scale steps.
        _generate("preview_pair", _grid(SIDES_13[:7]), L=4, H=16, n_seq=2, budget=1 / 10),
        # One 1024 x 1024 image pair at 20x compression, the benchmark's layer shape.
        _generate("image_pair_20x", full, L=4, H=16, n_seq=2, budget=1 / 20, bias=True),
        # Four image pairs at 10x; activations as a model's QKV projection leaves them, [sequence, token, head, d].
        _generate("batch8_10x", full, L=2, H=16, n_seq=8, budget=1 / 10, token_major=True),
        # A serving batch whose requests carry different budgets (budget 0: SERVING_BUDGETS in turn).
        _generate("serving_mixed", full, L=2, H=16, n_seq=16, budget=0.0),
        # The larger model's layer, 32 heads, batch 16: the largest launches.
        _generate("larger_20x", full, L=1, H=32, n_seq=16, budget=1 / 20, token_major=True),
        # The 8-bit cache.
        _generate("fp8_cache", full, L=2, H=16, n_seq=4, budget=1 / 10, cache="fp8"),
        # The dense per-head layout with in-place compaction, attention and cache update as two calls.
        _generate("ragged_5x", full, L=2, H=16, n_seq=4, budget=1 / 5, layout="ragged", fused=False),
        # Heads of 64 dimensions.
        _generate("heads_of_64", full, L=2, H=32, d=64, n_seq=2, budget=1 / 20),
        # Uncompressed cache, a 28-head layer, one image at an aspect ratio of 5 : 3 (odd, ragged token counts).
        _generate("uncompressed_5_3", _grid(SIDES_13, 5 / 3), L=2, H=28, n_seq=1, budget=1.0, fused=False),
        # Offline calibration from recorded activations, one call per layer.
        _calibrate("calibrate_recorded", full, L=1, H=16, n_seq=2, calls="recorded", bias=True),
        # Calibration while the model runs: every step's attention output goes on into the model.
        _calibrate("calibrate_forward", full, L=1, H=16, n_seq=2, calls="forward"),
    ]


def _log_int(rng, lo, hi):
    return min(hi, int(math.exp(rng.uniform(math.log(lo), math.log(hi + 1)))))


def draw(rng):
    while True:
        aspect = rng.choice((1.0, 1.0, 3 / 4, 4 / 3, 5 / 3, 9 / 16, 2.0))
        scales = _grid(SIDES_13[: rng.randint(4, 13)], aspect)
        c = dict(kind="generate", scales=scales, L=rng.randint(1, 4), H=_log_int(rng, 2, 40), d=rng.choice((64, 128, 128)),
                 n_seq=_log_int(rng, 1, 24), sinks=rng.choice((1, 2, SINKS)), bias=rng.random() < 0.3,
                 token_major=rng.random() < 0.5)
        if rng.random() < 0.25:
            c.update(kind="calibrate", calls=rng.choice(("recorded", "forward", "steps", "static")), L=min(c["L"], 2))
        else:
            c.update(budget=rng.choice((0.0, 1.0, math.exp(rng.uniform(math.log(1 / 40), 0.0)))),
                     cache=rng.choice(("bf16", "bf16", "fp8")), layout="paged", fused=rng.random() < 0.6)
            if c["cache"] == "bf16" and rng.random() < 0.25:
                c["layout"] = "ragged"
        t = _tokens(c)
        # the arrays of one state, in bytes: within what the largest listed case holds
        held = 8.0 * c["n_seq"] * c["H"] * c["d"] * sum(t) * c["L"]
        ctas = sum((x + 63) // 64 for x in t[-1:]) * c["H"] * c["n_seq"]
        if c.get("calls") == "static" and ctas > 16384:             # beyond that entry point's stated limit
            continue
        if held <= 6e9 and work(c)["flops"] <= MAX_FLOPS:
            return c


def _config(case):
    return hk.Config.make(case["L"], case["H"], case["d"], _tokens(case), case["sinks"])


def _scores(case):
    """S-CAS of the model: a log-normal strength per head, modulated per source scale."""
    rng = np.random.default_rng(20605)
    L, H, K = case["L"], case["H"], len(_tokens(case))
    return np.exp(rng.standard_normal((L, H, 1)) + 0.5 * rng.standard_normal((L, H, K))) / K


def _schedules(case):
    """One eviction schedule per sequence of the batch (sequences of equal budget share one)."""
    cfg, t = _config(case), _tokens(case)
    if case["budget"] < 0:
        fractions = np.resize(np.array((1.0, 0.5, 0.25, 0.0)), (case["L"], case["H"]))
        return [hk.heatkv_build_schedule(cfg, policy=hk.POLICY_EXPLICIT, fraction=fractions)] * case["n_seq"]
    # a short scale list cannot be compressed below its sinks
    least = min(1.0, 1.5 * sum(t[: case["sinks"]]) / max(1, sum(t[:-1])))
    budgets = [max(least, b) for b in (SERVING_BUDGETS if case["budget"] == 0 else (case["budget"],))]
    made = {b: hk.heatkv_build_schedule(cfg, scas=_scores(case), b=b) for b in set(budgets)}
    return [made[budgets[i % len(budgets)]] for i in range(case["n_seq"])]


class _State:
    """Context, schedules and activations of one program."""

    def __init__(self, case, seed):
        self.case, self.t = case, _tokens(case)
        self.L, self.H, self.n_seq, self.d = case["L"], case["H"], case["n_seq"], case["d"]
        self.schedules, self.session = [], None
        gen = torch.Generator(device="cuda").manual_seed(seed)
        tokens = sum(self.t)

        def activations():
            if case["token_major"]:
                x = torch.empty(self.n_seq, tokens, self.H, self.d, dtype=torch.bfloat16, device="cuda").transpose(1, 2)
            else:
                x = torch.empty(self.n_seq, self.H, tokens, self.d, dtype=torch.bfloat16, device="cuda")
            return x

        self.qkv = [tuple(activations().normal_(generator=gen) for _ in range(3)) for _ in range(self.L)]
        self.bias = None
        if case["bias"]:
            # heads differ in how far they look back: a logit offset on the current scale's own keys
            K = len(self.t)
            a = 4.0 * torch.rand(self.L, 1, self.H, 1, generator=gen, device="cuda")
            self.bias = (torch.eye(K, device="cuda").view(1, K, 1, K) * a).contiguous()       # [layer, step, head, scale]
        needs_out = case["kind"] == "generate" or case["calls"] == "forward"
        self.out = [activations() for _ in range(self.L)] if needs_out else []
        if case["kind"] == "generate":
            self.schedules = _schedules(case)
            layout = hk.LAYOUT_RAGGED if case["layout"] == "ragged" else hk.LAYOUT_PAGED
            fp8 = case["cache"] == "fp8"
            rows = stage = 0
            for s in self.schedules:
                rows += hk.heatkv_schedule_footprint(s, layout)[1]
                if fp8:
                    stage += max(64, hk.heatkv_schedule_plan_fp8(s)[1]) * self.d * 4
            self.session = Session(self.L, self.H, self.d, self.t, case["sinks"], pool_rows=rows, layout=layout,
                                   cache_dtype=hk.CACHE_FP8_E4M3 if fp8 else hk.CACHE_BF16, stage_bytes=stage)
        else:
            self.session = Session(self.L, self.H, self.d, self.t, case["sinks"], pool_rows=64)
            self.beta = torch.zeros(self.L, self.H, len(self.t), len(self.t), device="cuda")

    def __del__(self):
        if self.session is None or torch is None:
            return
        self.session.close()
        for s in set(self.schedules):
            hk.heatkv_schedule_free(s)


def prepare(case, seed):
    return _State(case, seed)


def run(state):
    if state.case["kind"] == "generate":
        return _run_generate(state)
    return _run_calibrate(state)


def _run_generate(state):
    ses = state.session
    ids = [hk.heatkv_seq_open(ses.ctx, s) for s in state.schedules]
    bias = state.bias
    ses.generate(ids, lambda layer: state.qkv[layer], lambda layer: state.out[layer],
                 None if bias is None else lambda layer, step: bias[layer, step], fused=state.case["fused"])
    for i in ids:
        hk.heatkv_seq_close(ses.ctx, i)
    return state.out


def _run_calibrate(state):
    ses, calls, n_seq = state.session, state.case["calls"], state.n_seq
    state.beta.zero_()
    for layer in range(state.L):
        q, k, v = state.qkv[layer]
        if calls == "recorded":
            hk.heatkv_calibrate_scores_steps(ses.ctx, layer, 0, ses.K, n_seq, q, k, hk.Strides.of(q, k),
                                             None if state.bias is None else state.bias[layer], state.beta)
            continue
        for step in range(ses.K):
            lo, hi = ses.step_slices(step)
            qs, ks = q[:, :, lo:hi], k[:, :, :hi]
            bias = None if state.bias is None else state.bias[layer, step]
            if calls == "forward":
                out = state.out[layer][:, :, lo:hi]
                hk.heatkv_calibrate_scores(ses.ctx, layer, step, n_seq, qs, ks, v[:, :, :hi], hk.Strides.of(qs, ks, out),
                                           bias, state.beta, out)
            elif calls == "steps":
                hk.heatkv_calibrate_scores(ses.ctx, layer, step, n_seq, qs, ks, None, hk.Strides.of(qs, ks), bias,
                                           state.beta, None)
            else:
                hk.heatkv_calibrate_scores_static(ses.ctx, layer, step, n_seq, qs, ks, hk.Strides.of(qs, ks), bias,
                                                  state.beta)
    return [state.beta] + state.out


def work(case):
    """Q, K, V of every step in and its output out once, every visible cached row in and every stored row out once;
    2 d operations per (query, key) pair for the scores and 2 d for the output."""
    t, L, H, d, n_seq = _tokens(case), case["L"], case["H"], case["d"], case["n_seq"]
    K, own = len(t), float(sum(t))
    if case["kind"] == "calibrate":
        pairs = float(sum(t[k] * sum(t[: k + 1]) for k in range(K)))
        out = case["calls"] == "forward"
        return {"bytes": n_seq * L * H * own * d * 2.0 * (4 if out else 2) + L * H * K * (K + 1) / 2 * 4.0,
                "flops": n_seq * L * H * pairs * d * (4.0 if out else 2.0)}
    flops = bytes_ = 0.0
    row = 2.0 * (d + 1 if case["cache"] == "fp8" else 2 * d)       # a cached row, K and V
    schedules = _schedules(case)
    tokens = np.array(t, dtype=np.float64)
    bits = 1 << np.arange(K)
    for sch in set(schedules):
        attn, keep = hk.heatkv_schedule_masks(sch, K, L, H)[:2]
        visible = ((attn[..., None].astype(np.int64) & bits) != 0) @ tokens          # [step, layer, head]
        for k in range(K):
            stored = ((keep[k] >> k) & 1).sum() * t[k] if k + 1 < K else 0
            n = schedules.count(sch)
            flops += n * 4.0 * d * t[k] * float((visible[k] + t[k]).sum())
            bytes_ += n * (L * H * t[k] * 8.0 * d + float(visible[k].sum()) * row + stored * row)
    for sch in set(schedules):
        hk.heatkv_schedule_free(sch)
    return {"bytes": bytes_, "flops": flops}


def tolerance(case):
    """Measured against a 64-bit computation, times four: bf16 outputs from bf16 probabilities are off by 2.0e-3 to 2.1e-3
    of their norm and by at most 0.043 of their root mean square.  The mass per source scale, a 32-bit sum, came within
    2e-7; 1e-5 leaves room for sums in another order over more sequences."""
    if case["kind"] == "calibrate" and case["calls"] != "forward":
        return {"rel": 1e-5, "max": 1e-4}
    return {"rel": 8e-3, "max": 0.17}
