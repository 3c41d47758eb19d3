"""Blocks of at most 32 tokens: a warp works off all tensors of a (head, block), or, where there are fewer of those than warps, one
tensor of it.  Both give the same maps and the same merged tensors, bit for bit."""
import numpy as np
import pytest
import torch

from paper_2511_21317_b200 import binding as hb
from paper_2511_21317_b200 import synth
from tests.test_gpu_parity import run_case

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
ITEMS = {"assign_q": hb.X_ASSIGN_Q, "assign_k": hb.X_ASSIGN_K, "rank_q": hb.X_RANK_Q, "q_m": hb.X_Q_MERGED, "k_m": hb.X_K_MERGED, "v_m": hb.X_V_MERGED}


def run(cfg, qkv):
    with hb.Httm(cfg) as ctx:
        ctx.global_attention(*qkv)
        torch.cuda.synchronize()
        assert ctx.query(hb.Q_DEVICE_STATUS) == 0
        return {n: ctx.export(w) for n, w in ITEMS.items()}


@pytest.mark.parametrize("blk,ratio,specials,frames", [((2, 4, 4), 0.7, 4, 12), ((1, 3, 5), 0.5, 0, 12), ((3, 3, 3), 0.9, 2, 13), ((2, 4, 4), 0.6, 40, 12),
                                                       ((2, 2, 8), 0.0, 1, 12), ((3, 3, 3), 0.7, 2, 13)],
                         ids=["32_tokens", "15_tokens", "27_tokens", "over_reordered_copies", "keys_only", "equal_ratios"])
def test_whole_units_and_split_units_agree(blk, ratio, specials, frames):
    """24 heads have more units than the chip has warps for, one head has fewer."""
    wl = synth.Workload("units", frames, 22, 25, *blk, ratio, 0.7, n_camera=1, n_register=specials, heads=24, seed=2)
    q, k, v = (hb.bf16_from_bits(x, DEV) for x in synth.make_qkv(wl))
    whole = run(hb.HttmConfig.of(wl), (q, k, v))
    for h in (0, 11, 23):
        one = run(hb.HttmConfig.of(wl.replace(heads=1)), (q[h:h + 1], k[h:h + 1], v[h:h + 1]))
        for name in ITEMS:
            assert np.array_equal(whole[name][h], one[name][0]), (name, h)


@pytest.mark.parametrize("blk,frames,columns", [((1, 4, 8), 3, 37), ((1, 4, 8), 3, 38), ((1, 4, 16), 2, 37), ((1, 4, 16), 2, 38)],
                         ids=["32_as_many_as_warps", "32_more", "64_as_many_as_warps", "64_more"])
@pytest.mark.parametrize("specials", [4, 44], ids=["direct", "over_reordered_copies"])
def test_as_many_tensors_of_blocks_as_warps(blk, frames, columns, specials):
    """One tensor for each warp that fits on the chip (24 or 16 of them on each of 148 SMs), and a few more than that, against the same heads alone."""
    wl = synth.Workload("limit", frames, 4, columns * blk[2], *blk, 0.5, 0.7, n_camera=1, n_register=specials, heads=16, seed=5)
    tensors, warps = 2 * wl.heads * frames * columns, (24 if blk[2] == 8 else 16) * 148
    assert (tensors == warps) == (columns == 37) and tensors >= warps
    q, k, v = (hb.bf16_from_bits(x, DEV) for x in synth.make_qkv(wl))
    whole = run(hb.HttmConfig.of(wl), (q, k, v))
    for h in (0, 7, 15):
        one = run(hb.HttmConfig.of(wl.replace(heads=1)), (q[h:h + 1], k[h:h + 1], v[h:h + 1]))
        for name in ITEMS:
            assert np.array_equal(whole[name][h], one[name][0]), (name, h)


@pytest.mark.parametrize("blk,ratio", [((2, 4, 4), 0.04), ((2, 4, 4), 0.46), ((2, 4, 4), 0.5), ((2, 4, 4), 0.53), ((2, 4, 4), 0.97), ((1, 4, 4), 0.07), ((1, 4, 4), 0.94),
                                       ((1, 1, 17), 0.06), ((3, 3, 3), 0.4), ((1, 1, 2), 0.5)])
def test_numbers_of_kept_rows_and_tokens(blk, ratio):
    """One and two 16-row tiles of merged rows (31, 18, 16, 15 and 1 kept of 32 tokens), one and two 16-token steps (15 and 1 kept of 16, 16 of 17), against the
    oracle; the blocks at the edges of the grid are clipped."""
    wl = synth.Workload("kept", 5, 9, 18, *blk, ratio, ratio, n_camera=1, n_register=2, heads=2, seed=7)
    stats = run_case(wl, peaky=True)
    assert stats["peaky_needed"] <= 0.001 * stats["out_elements"]


@pytest.mark.parametrize("ratio", [0.0, 0.5, 0.72, 0.75, 0.8, 0.97])
@pytest.mark.parametrize("strided", [False, True])
def test_rows_with_many_target_tokens(ratio, strided):
    """The epilogue that unmerges stores 32 rows to all their target tokens, 128 targets at a time: one target per row up to 32, lists just
    below and above 128, 256 and more, tiles whose last rows do not exist, rows of a wider output too.  The same rows through the unmerge kernel."""
    wl = synth.Workload("targets", 8, 20, 24, 2, 4, 4, ratio, 0.5, n_camera=1, n_register=2, heads=3, seed=6)
    q, k, v = (hb.bf16_from_bits(x, DEV) for x in synth.make_qkv(wl))
    n = wl.n_tokens
    with hb.Httm(hb.HttmConfig.of(wl)) as ctx:
        wide = wl.heads * 64 + (72 if strided else 0)   # (rows of a wider tensor)
        outs = [torch.zeros(n, wide, dtype=torch.bfloat16, device=DEV)[:, :wl.heads * 64] for _ in range(2)]
        ctx.global_attention(q, k, v, outs[0])
        ctx.launch_stage(hb.STAGE_ATTENTION)
        ctx.launch_stage(hb.STAGE_UNMERGE, out=outs[1])
        torch.cuda.synchronize()
        assert ctx.query(hb.Q_DEVICE_STATUS) == 0
        assert torch.equal(outs[0], outs[1])
