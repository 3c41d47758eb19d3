"""The work a program has this library do, as cases that can be timed and compared.

A case is one pass through the public entry points (`paper_2511_21317_b200.binding`): an HTTM global-attention layer on
device tensors, the same layer with its projections, on host buffers, the unmerged (dense) layer, or a projection alone.
Geometries are those of `synth.WORKLOADS` and of the benchmark's sweep, and ragged ones like the tests'.  Inputs are the
correlated field of `synth` (a smooth periodic field that drifts by one patch per frame, plus noise; N(0, 1) special
tokens), drawn on the GPU.
"""
from __future__ import annotations

import math

import torch

from paper_2511_21317_b200 import binding as hb

_LATTICE = 8
_HEAD_DIM = 64
_SPECIAL = 5          # one camera token and four registers per frame
_MAX_FLOPS = 4.4e12   # of a drawn case: below the largest listed one
_MAX_TOKENS = 137400


def _case(name, op, frames, grid, block, ratio_q, ratio_kv, **kw):
    c = {"name": name, "op": op, "frames": frames, "grid_h": grid[0], "grid_w": grid[1], "blk_frames": block[0], "blk_h": block[1],
         "blk_w": block[2], "ratio_q": ratio_q, "ratio_kv": ratio_kv, "heads": 16, "outliers": 0.0, "anchor": 0, "sigma": 0.1,
         "layout": "heads", "field_h": grid[0], "field_w": grid[1]}
    c.update(kw)
    return c


def listed():
    return [
        # A pair of small images (the "tiny" workload), Q / K / V as views of the fused projection output, as a network hands them
        # over: launches and latency count.
        _case("tiny", "merged", 4, (16, 16), (2, 4, 4), 0.5, 0.5, layout="fused"),
        # A short sequence at VGGT's 37 x 37 patches ("small"): the query tiles do not fill the chip evenly.
        _case("small", "merged", 8, (37, 37), (2, 4, 4), 0.7, 0.7),
        # The benchmark's workload.
        _case("medium", "merged", 24, (37, 37), (2, 4, 4), 0.7, 0.7),
        # The same scene with the adaptive outlier filtering of the queries (Sec. 3.4).
        _case("medium_outliers", "merged", 24, (37, 37), (2, 4, 4), 0.7, 0.7, outliers=0.01, layout="fused"),
        # Wide windows and a high ratio, a point of the benchmark's sweep: 128-token blocks, the merging weighs as much as the attention.
        _case("windows_2x8x8", "merged", 24, (37, 37), (2, 8, 8), 0.9, 0.9, layout="fused"),
        # A ragged scene (clipped blocks in every direction) with the first frame as the reference frame (the paper's appendix).
        _case("ragged_anchored", "merged", 11, (23, 31), (3, 4, 4), 0.6, 0.6, anchor=1, layout="fused"),
        # A long sequence with noisier features ("large").
        _case("large", "merged", 100, (37, 37), (4, 4, 4), 0.8, 0.8, sigma=0.3),
        # The paper's own configuration: runs of 128 patches over 30 frames, 90 % / 70 % merged, 10 % outliers (Sec. 4.1).
        _case("paper_1d_outliers", "merged", 60, (1, 1369), (30, 1, 128), 0.9, 0.7, outliers=0.1, field_h=37, field_w=37),
        # One layer of the 24-layer stack: QKV projection, HTTM attention on views of its output, output projection.
        _case("stack_layer", "layer", 48, (37, 37), (2, 4, 4), 0.7, 0.7, layout="fused"),
        # The unmerged layer the speed-ups are quoted against; also what a program runs in the layers it does not merge.
        _case("dense_medium", "dense", 24, (37, 37), (2, 4, 4), 0.7, 0.7),
        # The QKV projection of a short sequence.
        _case("qkv_projection", "linear", 8, (37, 37), (2, 4, 4), 0.7, 0.7),
        # The layer for a caller whose tensors are in (pinned) host memory.
        _case("small_host", "host", 8, (37, 37), (2, 4, 4), 0.7, 0.7),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: 2 .. 100 frames of 8 .. 40 patches a side (odd and unequal sides among them), the block shapes and ratios of
    the sweep, long runs as in the paper, both layouts, both options."""
    while True:
        op = rng.choice(["merged"] * 8 + ["layer", "layer", "dense", "linear", "host"])
        frames, gh, gw = _log_int(rng, 2, 100), rng.randint(8, 40), rng.randint(8, 40)
        ratio_q = round(rng.uniform(0.5, 0.9), 2)
        ratio_kv = ratio_q if rng.random() < 0.7 else round(rng.uniform(0.5, 0.9), 2)
        runs = op == "merged" and rng.random() < 0.15
        if runs:   # a frame handed over as one run of patches; blocks of up to 30 frames
            grid, block, field = (1, gh * gw), (min(frames, rng.randint(8, 30)), 1, rng.choice([64, 96, 128])), (gh, gw)
        else:
            grid, field = (gh, gw), (gh, gw)
            block = rng.choice([(2, 4, 4), (2, 4, 4), (2, 4, 4), (4, 4, 4), (2, 8, 8), (1, 4, 4), (3, 4, 4), (2, 3, 5)])
        c = _case("", op, frames, grid, block, ratio_q, ratio_kv, heads=rng.choice([16, 16, 16, 8]), sigma=rng.choice([0.1, 0.1, 0.3]),
                  layout="fused" if op == "layer" or (op == "merged" and rng.random() < 0.5) else "heads", field_h=field[0], field_w=field[1])
        if op == "merged":
            c["outliers"] = rng.choice([0.0, 0.0, 0.0, 0.01, 0.1])
            c["anchor"] = 1 if not runs and rng.random() < 0.15 else 0
        del c["name"]
        if _tokens(c) <= _MAX_TOKENS and work(c)["flops"] <= _MAX_FLOPS:
            return c


def _tokens(c):
    return c["frames"] * (_SPECIAL + c["grid_h"] * c["grid_w"])


def _pieces(total, size):
    """Lengths of the pieces a side is cut into (the last one may be clipped)."""
    return [min(size, total - i) for i in range(0, total, size)]


def _merged_counts(c):
    """(merged queries, merged keys, multiply-adds of the similarities) of one head."""
    n_tok = _tokens(c)
    m, macs = [n_tok, n_tok], 0
    for g, bt in enumerate(_pieces(c["frames"], c["blk_frames"])):
        for bh in _pieces(c["grid_h"], c["blk_h"]):
            for bw in _pieces(c["grid_w"], c["blk_w"]):
                n = bt * bh * bw
                for t, ratio in enumerate((c["ratio_q"], c["ratio_kv"])):
                    if c["anchor"] and g == 0:
                        dst = bh * bw
                        r = min(int(ratio * n + 1e-9), n - dst)
                    else:
                        r = min(int(ratio * n + 1e-9), n - 1)
                        dst = min(-(-n // 4), n - r)
                    m[t] -= r
                    macs += (n - dst) * dst * _HEAD_DIM if r > 0 else 0
    return m[0], m[1], macs


def work(case):
    n, h = _tokens(case), case["heads"]
    dim = h * _HEAD_DIM
    if case["op"] == "linear":
        return {"bytes": 2.0 * (n * dim + 3 * dim * dim + n * 3 * dim), "flops": 2.0 * n * dim * 3 * dim}
    if case["op"] == "dense":
        return {"bytes": 2.0 * 4 * n * dim, "flops": 4.0 * dim * n * n}
    mq, mk, macs = _merged_counts(case)
    queries = h * mq + min(math.floor(case["outliers"] * h * n + 1e-9), h * (n - mq))
    flops = 4.0 * _HEAD_DIM * queries * mk + 2.0 * h * macs
    if case["op"] == "layer":   # x -> y, and both weights; Q, K, V and the attention output are intermediates
        return {"bytes": 2.0 * (2 * n * dim + 4 * dim * dim), "flops": flops + 2.0 * n * dim * 4 * dim}
    return {"bytes": 2.0 * 4 * n * dim, "flops": flops}


def tolerance(case):
    """bf16 inputs, weights and outputs with fp32 accumulation: against the same path in 64 bits (merged as the kernels merge) the
    outputs of every kind of case are off by 1.7e-3 (2-norm), the largest element by 0.004 (dense, projection) and 0.007 (merged);
    four times that is allowed.  The largest difference of a merged layer is left wide: where two partners of a token are equally
    similar within the rounding of the similarity (fp32), another correct implementation may merge it into the other one, and the
    outputs of the few tokens of that block then differ by as much as the outputs themselves."""
    return {"rel": 7e-3, "max": 0.016 if case["op"] in ("linear", "dense") else 0.9}


def _field(c, gen):
    """One tensor [heads][tokens][64], bf16: the smooth field, drifting by one patch per frame, plus noise; random special tokens."""
    H, S, fh, fw, dev = c["heads"], c["frames"], c["field_h"], c["field_w"], gen.device
    lattice = torch.randn(H, _LATTICE, _LATTICE, _HEAD_DIM, generator=gen, device=dev)
    y = torch.arange(fh, device=dev) * (_LATTICE / fh)
    x = torch.arange(fw, device=dev) * (_LATTICE / fw)
    y0, x0 = y.floor().long(), x.floor().long()
    fy, fx = (y - y0).view(1, fh, 1, 1), (x - x0).view(1, 1, fw, 1)
    y1, x1 = (y0 + 1) % _LATTICE, (x0 + 1) % _LATTICE
    rows = lattice[:, y0] * (1 - fy) + lattice[:, y1] * fy
    smooth = rows[:, :, x0] * (1 - fx) + rows[:, :, x1] * fx                                     # [H][fh][fw][64]
    at = (torch.arange(fw, device=dev).view(1, fw) + torch.arange(S, device=dev).view(S, 1)) % fw    # column seen by (frame, x)
    out = torch.empty(H, S, _SPECIAL + fh * fw, _HEAD_DIM, dtype=torch.bfloat16, device=dev)
    for h in range(H):
        noise = torch.randn(S, _SPECIAL + fh * fw, _HEAD_DIM, generator=gen, device=dev)
        out[h, :, :_SPECIAL] = noise[:, :_SPECIAL]
        seen = smooth[h][:, at].permute(1, 0, 2, 3).reshape(S, fh * fw, _HEAD_DIM)
        out[h, :, _SPECIAL:] = seen + c["sigma"] * noise[:, _SPECIAL:]
    return out.view(H, S * (_SPECIAL + fh * fw), _HEAD_DIM)


def prepare(case, seed):
    device = "cuda:0"
    gen = torch.Generator(device=device).manual_seed(seed)
    n, h = _tokens(case), case["heads"]
    dim = h * _HEAD_DIM
    ctx = hb.Httm(hb.HttmConfig(frames=case["frames"], grid_h=case["grid_h"], grid_w=case["grid_w"], blk_frames=case["blk_frames"],
                                blk_h=case["blk_h"], blk_w=case["blk_w"], ratio_q=case["ratio_q"], ratio_kv=case["ratio_kv"],
                                heads=h, anchor_first_frame=case["anchor"]))
    if case["outliers"] > 0:
        ctx.set_outlier_fraction(case["outliers"])
    st = {"op": case["op"], "ctx": ctx}
    if case["op"] in ("linear", "layer"):
        st["x"] = _field(case, gen).permute(1, 0, 2).reshape(n, dim).contiguous()
        st["w_qkv"] = (torch.randn(3 * dim, dim, generator=gen, device=device) * 0.02).to(torch.bfloat16)
        st["qkv"] = torch.empty(n, 3 * dim, dtype=torch.bfloat16, device=device)
    if case["op"] == "layer":
        st["w_o"] = (torch.randn(dim, dim, generator=gen, device=device) * 0.02).to(torch.bfloat16)
        st["attn"] = torch.empty(n, dim, dtype=torch.bfloat16, device=device)
        st["y"] = torch.empty(n, dim, dtype=torch.bfloat16, device=device)
        views = st["qkv"].view(n, 3, h, _HEAD_DIM)
        st["q"], st["k"], st["v"] = (views[:, i].permute(1, 0, 2) for i in range(3))
    elif case["op"] != "linear":
        q, k, v = (_field(case, gen) for _ in range(3))
        if case["layout"] == "fused":   # views of one [tokens][3][heads][64] tensor
            fused = torch.empty(n, 3, h, _HEAD_DIM, dtype=torch.bfloat16, device=device)
            for i, t in enumerate((q, k, v)):
                fused[:, i] = t.permute(1, 0, 2)
            q, k, v = (fused[:, i].permute(1, 0, 2) for i in range(3))
        st["out"] = torch.empty(n, dim, dtype=torch.bfloat16, device=device)
        if case["op"] == "host":
            q, k, v = (t.cpu().pin_memory() for t in (q, k, v))
            st["out"] = torch.empty(n, dim, dtype=torch.bfloat16, pin_memory=True)
        st["q"], st["k"], st["v"] = q, k, v
    return st


def run(state):
    ctx, op = state["ctx"], state["op"]
    if op == "linear":
        return ctx.linear(state["x"], state["w_qkv"], state["qkv"])
    if op == "layer":
        ctx.linear(state["x"], state["w_qkv"], state["qkv"])
        ctx.global_attention(state["q"], state["k"], state["v"], state["attn"])
        return ctx.linear(state["attn"], state["w_o"], state["y"])
    if op == "dense":
        return ctx.dense_attention(state["q"], state["k"], state["v"], state["out"])
    if op == "host":   # asynchronous: `out` may be read once the stream has been synchronised
        return ctx.attention_host(state["q"], state["k"], state["v"], state["out"])
    return ctx.global_attention(state["q"], state["k"], state["v"], state["out"])
