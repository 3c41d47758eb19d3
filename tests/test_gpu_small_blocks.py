"""Blocks of at most 32 tokens: a warp works off all tensors of a (head, block), or, where there are fewer of those than warps, one
tensor of it.  Both give the same maps and the same merged tensors, bit for bit."""
import numpy as np
import pytest
import torch

from paper_2511_21317_b200 import binding as hb
from paper_2511_21317_b200 import synth

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
