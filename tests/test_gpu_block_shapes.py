"""Merge maps of scenes whose clipped blocks come in several shapes of the same token count, against the oracle.

The match kernels keep what follows from a block's shape (stage rows of its dst tokens, token numbers of its rows) from block to block and
make it anew when the shape changes.  With blk_frames == blk_w and the same remainder of the frames and of the patch columns, a block
clipped in time and one clipped in width have equally many tokens and dst tokens: only the shape itself tells them apart.  Equal ratios for
queries and keys (with other ratios the tables are made anew for every tensor), and more blocks than warps or teams."""
import numpy as np
import pytest
import torch

from oracle import httm_oracle as orc
from paper_2511_21317_b200 import binding as hb
from paper_2511_21317_b200 import synth
from tests import parity

pytestmark = pytest.mark.gpu

# (block, frames, grid_h, grid_w, ratio, heads)
SCENES = {
    "2x2x2": ((2, 2, 2), 5, 41, 41, 0.5, 12),          # one warp per block
    "3x3x3": ((3, 3, 3), 13, 22, 25, 0.7, 24),
    "4x2x4": ((4, 2, 4), 13, 22, 25, 0.6, 24),
    "4x4x4": ((4, 4, 4), 9, 37, 37, 0.7, 16),          # teams for blocks of up to 64, 128 and 256 tokens
    "4x4x4_remainder_2": ((4, 4, 4), 50, 22, 30, 0.7, 16),
    "6x3x6": ((6, 3, 6), 13, 25, 25, 0.7, 8),
    "8x4x8": ((8, 4, 8), 13, 25, 37, 0.7, 16),
}


@pytest.mark.parametrize("name", sorted(SCENES))
def test_maps_where_clipped_blocks_have_the_same_size(name):
    blk, frames, grid_h, grid_w, ratio, heads = SCENES[name]
    assert blk[0] == blk[2] and frames % blk[0] == grid_w % blk[2] != 0
    wl = synth.Workload(name, frames, grid_h, grid_w, *blk, ratio, ratio, heads=heads, seed=4)
    q, k, v = synth.make_qkv(wl)
    with hb.Httm(hb.HttmConfig.of(wl)) as ctx:
        ctx.global_attention(*(hb.bf16_from_bits(x, "cuda:0") for x in (q, k, v)))
        torch.cuda.synchronize()
        assert ctx.query(hb.Q_DEVICE_STATUS) == 0
        maps = ctx.export(hb.X_ASSIGN_Q), ctx.export(hb.X_ASSIGN_K)
    g = orc.Geometry.of(wl)
    res = orc.global_attention(g, ratio, ratio, q, k, v, attend=False)
    parity.check_maps(g, ratio, res.blk_start, orc.reorder(g, res.pi, q), res.assign_q, res.margin_best_q, res.margin_sel_q, maps[0], name + " A_q")
    parity.check_maps(g, ratio, res.blk_start, orc.reorder(g, res.pi, k), res.assign_k, res.margin_best_k, res.margin_sel_k, maps[1], name + " A_k")
