"""Attention with query tiles that are split over CTAs: where a few 128-row query tiles are left after whole tiles have been dealt,
each of them is worked off in parts of its keys by several CTAs; of the warps with the same rows the one that arrives last adds the partial softmaxes up."""
import pytest
import torch

from paper_2511_21317_b200 import binding as hb
from paper_2511_21317_b200 import synth
from tests import parity

pytestmark = pytest.mark.gpu
DEV = "cuda:0"

# (heads, frames, blocks, ratio_q, ratio_kv, outlier fraction): tiles left, and parts, on 148 SMs
CASES = {
    "few_tiles": (2, 4, (2, 4, 4), 0.9, 0.0, 0.0),            # 12 tiles in 5 parts of 8 or 9 key tiles, unmerge in the epilogue
    "one_head_many_parts": (1, 11, (4, 4, 4), 0.9, 0.0, 0.0),  # 14 tiles in 10 parts of 11 or 12, plain rows
    "two_parts": (12, 4, (2, 4, 4), 0.9, 0.0, 0.0),            # 72 tiles in 2 parts of 21 or 22
    "singles_then_parts": (16, 8, (2, 4, 4), 0.7, 0.4, 0.0),   # 448 tiles: a round of pairs, one of single tiles, 4 tiles in 6 parts
    "per_head_lengths": (2, 8, (2, 4, 4), 0.8, 0.2, 0.03),     # the plan is made on the device
}


def reference(q, k, v):
    return torch.softmax((q.double() @ k.double().T) / 8, -1) @ v.double()


@pytest.mark.parametrize("jump", [False, True], ids=["plain", "scores_jump"])
@pytest.mark.parametrize("name", sorted(CASES))
def test_split_tiles(name, jump):
    """Against the same merged tensors in 64 bits, within the tolerance of the attention output, and the same bits again.
    scores_jump: keys of the last frames score more than 2^100 above the others, so the maxima of a tile's parts differ by that much
    and the tile that meets them is redone."""
    heads, frames, blk, rq, rkv, gamma = CASES[name]
    wl = synth.Workload(name, frames, 37, 37, *blk, rq, rkv, heads=heads, seed=3)
    q, k, v = (hb.bf16_from_bits(x, DEV) for x in synth.make_qkv(wl))
    if jump:
        q[..., 0] = 8.0
        k[..., 0] = 0.0
        k[:, -2 * wl.tokens_per_frame:, 0] = 80.0
    with hb.Httm(hb.HttmConfig.of(wl)) as ctx:
        ctx.set_outlier_fraction(gamma)
        out = ctx.global_attention(q, k, v)
        torch.cuda.synchronize()
        assert ctx.query(hb.Q_DEVICE_STATUS) == 0
        again = ctx.global_attention(q, k, v)
        torch.cuda.synchronize()
        assert torch.equal(out, again)
        m = {n: hb.bf16_from_bits(ctx.export(w), DEV) for n, w in (("q", hb.X_Q_MERGED), ("k", hb.X_K_MERGED), ("v", hb.X_V_MERGED))}
        rank, pi_inv = (torch.from_numpy(ctx.export(w)).to(DEV).long() for w in (hb.X_RANK_Q, hb.X_PI_INV))
        lens = ctx.export(hb.X_MERGED_Q_HEAD) if gamma else [ctx.m_q] * heads
    for h in range(heads):
        ref = reference(m["q"][h][:int(lens[h])], m["k"][h], m["v"][h])[rank[h][pi_inv]]
        got = out[:, 64 * h:64 * h + 64].double()
        err = (got - ref).abs().max() / ref.pow(2).mean().sqrt()
        assert err <= parity.OUT_TOL, (name, h, float(err))


# (heads, tokens): query tiles per head, unpaired ones, and how they are dealt on 148 SMs
ODD = {
    "one_tile_each": (200, 100),               # no pairs at all: two single tiles per CTA
    "own_ctas": (60, 300),                     # 3 tiles: 60 pairs and 60 unpaired tiles in one partial round
    "two_per_cta": (98, 300),                  # 3 tiles: 98 pairs, the 98 unpaired tiles two by two on the CTAs that are left
    "unpaired_after_full_rounds": (75, 600),   # 5 tiles: 148 pairs, then the other 4 tiles and the 75 unpaired ones on CTAs of their own
    "even": (75, 500),                         # 4 tiles: nothing unpaired
}


@pytest.mark.parametrize("name", sorted(ODD))
def test_heads_with_an_odd_number_of_tiles(name):
    heads, tokens = ODD[name]
    gen = torch.Generator(device=DEV).manual_seed(7)
    q, k, v = (torch.randn(heads, tokens, 64, device=DEV, generator=gen).bfloat16() for _ in range(3))
    with hb.Httm(hb.HttmConfig(frames=1, n_camera=0, n_register=0, grid_h=10, grid_w=tokens // 10, heads=heads, head_dim=64, blk_frames=1, blk_h=2, blk_w=2,
                               ratio_q=0.5, ratio_kv=0.5)) as ctx:
        out = ctx.dense_attention(q, k, v)
        torch.cuda.synchronize()
        assert ctx.query(hb.Q_DEVICE_STATUS) == 0
    for h in range(heads):
        ref = reference(q[h], k[h], v[h])
        # few keys dominate some rows of random inputs, with values far above the RMS: the bf16 rounding of the output is allowed for
        err = (out[:, 64 * h:64 * h + 64].double() - ref).abs() - 2.0 ** -8 * ref.abs()
        assert err.max() <= parity.OUT_TOL * ref.pow(2).mean().sqrt(), (name, h, float(err.max()))
