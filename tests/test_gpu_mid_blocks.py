"""Blocks of 33 .. 256 tokens at the limits of the teams that work them off, against the oracle; and many blocks per team, where loads,
tables and groups run one block ahead, against the same head alone, bit for bit."""
import numpy as np
import pytest

from oracle import httm_oracle as orc
from paper_2511_21317_b200 import binding as hb
from paper_2511_21317_b200 import synth
from tests.test_gpu_parity import report_peaky, run_case
from tests.test_gpu_small_blocks import ITEMS, run

pytestmark = pytest.mark.gpu


# (block, ratio_q, ratio_kv): few merge (picked one by one), half, nearly all; block sizes around 32, 64, 128 and 256
@pytest.mark.parametrize("blk,ratio_q,ratio_kv", [((1, 3, 11), 0.1, 0.9), ((4, 4, 4), 0.375, 0.2), ((1, 5, 13), 0.1, 0.7), ((2, 8, 8), 0.4, 0.0),
                                                  ((3, 1, 43), 0.3, 0.95), ((4, 8, 8), 0.1, 0.5), ((3, 5, 17), 0.7, 0.99)],
                         ids=["33", "64", "65", "128", "129", "256", "255"])
def test_limits_of_the_teams(blk, ratio_q, ratio_kv):
    wl = synth.Workload("limits", 4, blk[1] + 4, 2 * blk[2] + 1, *blk, ratio_q, ratio_kv, n_camera=1, n_register=4, heads=2, seed=5)
    report_peaky("limits", run_case(wl, peaky=True))
    x = synth.make_identical_block_tokens(wl, seed=6)   # all similarities of a block are ties: the order of the positions decides
    _, k, v = synth.make_qkv(wl)
    report_peaky("ties", run_case(wl, x, x, v, peaky=True))


@pytest.mark.parametrize("blk,frames,specials", [((4, 4, 4), 34, 4), ((2, 8, 8), 41, 4), ((4, 8, 8), 42, 4), ((4, 4, 4), 34, 70)],
                         ids=["64", "128", "256", "over_reordered_copies"])
def test_many_blocks_per_team(blk, frames, specials):
    wl = synth.Workload("many", frames, 21, 26, *blk, 0.6, 0.8, n_camera=1, n_register=specials, heads=24, seed=2)
    q, k, v = (hb.bf16_from_bits(x, "cuda:0") for x in synth.make_qkv(wl))
    whole = run(hb.HttmConfig.of(wl), (q, k, v))
    for h in (0, 13, 23):
        one = run(hb.HttmConfig.of(wl.replace(heads=1)), (q[h:h + 1], k[h:h + 1], v[h:h + 1]))
        for name in ITEMS:
            assert np.array_equal(whole[name][h], one[name][0]), (name, h)


@pytest.mark.parametrize("blk,ratio_q,ratio_kv", [((1, 3, 11), 0.1, 0.95), ((3, 4, 4), 0.75, 0.0), ((3, 3, 5), 0.3, 0.86), ((1, 7, 7), 0.5, 0.9), ((4, 4, 4), 0.25, 0.97)],
                         ids=["33", "48", "45", "49", "64"])
def test_whole_units_and_split_units_of_33_to_64_tokens_agree(blk, ratio_q, ratio_kv):
    """Blocks of 33 .. 64 tokens go to one warp of the small-block kernel, several tensors of them in turn where there are many: few merge and nearly all, eight dst tokens
    and sixteen, clipped blocks, equal similarities.  Those of the same head alone go to a warp each."""
    wl = synth.Workload("many", 12 * blk[0] + 1, 5 * blk[1] + 2, 3 * blk[2] + 1, *blk, ratio_q, ratio_kv, n_camera=1, n_register=4, heads=16, seed=4)
    assert 13 * 6 * 4 * wl.heads > 16 * 148 >= 13 * 6 * 4   # (units against warps)
    q, k, v = synth.make_qkv(wl)
    q[3] = synth.make_identical_block_tokens(wl, seed=6)[3]
    q, k, v = (hb.bf16_from_bits(x, "cuda:0") for x in (q, k, v))
    whole = run(hb.HttmConfig.of(wl), (q, k, v))
    for h in (0, 3, 15):
        one = run(hb.HttmConfig.of(wl.replace(heads=1)), (q[h:h + 1], k[h:h + 1], v[h:h + 1]))
        for name in ITEMS:
            assert np.array_equal(whole[name][h], one[name][0]), (name, h)


@pytest.mark.parametrize("blk,ratio_q,ratio_kv", [((3, 4, 4), 0.75, 0.0), ((1, 7, 7), 0.5, 0.9), ((4, 4, 4), 0.25, 0.97)], ids=["48", "49", "64"])
def test_several_tensors_per_warp_and_one_agree(blk, ratio_q, ratio_kv):
    """The same with 24 heads: six or seven tensors in turn, those of Q first (with 16 heads five, dealt out evenly)."""
    wl = synth.Workload("many", 12 * blk[0] + 1, 5 * blk[1] + 2, 3 * blk[2] + 1, *blk, ratio_q, ratio_kv, n_camera=1, n_register=4, heads=24, seed=4)
    tasks, warps = 2 * 13 * 6 * 4 * wl.heads, 16 * 148
    assert -(-tasks // warps) == 7 and 2 * 13 * 6 * 4 <= warps
    q, k, v = synth.make_qkv(wl)
    q[3] = synth.make_identical_block_tokens(wl, seed=6)[3]
    q, k, v = (hb.bf16_from_bits(x, "cuda:0") for x in (q, k, v))
    whole = run(hb.HttmConfig.of(wl), (q, k, v))
    for h in (0, 3, 23):
        one = run(hb.HttmConfig.of(wl.replace(heads=1)), (q[h:h + 1], k[h:h + 1], v[h:h + 1]))
        for name in ITEMS:
            assert np.array_equal(whole[name][h], one[name][0]), (name, h)


@pytest.mark.parametrize("blk,ratio", [((2, 8, 8), 0.5), ((2, 8, 8), 0.7), ((1, 5, 13), 0.3), ((4, 8, 8), 0.6), ((4, 4, 4), 0.5), ((2, 4, 4), 0.5), ((2, 4, 4), 0.3)])
def test_some_scores_are_equal(blk, ratio):
    """Tokens that are one of a few vectors: the line between those that merge and the others runs through scores that are equal but for their rounding."""
    wl = synth.Workload("equal", 3, blk[1] + 3, 2 * blk[2] + 1, *blk, ratio, ratio, n_camera=1, n_register=1, heads=3, seed=8)
    q, k, v = synth.make_qkv(wl)
    rng = np.random.default_rng(9)
    for h in range(wl.heads):
        kinds = q[h, rng.integers(0, wl.n_tokens, size=3 + 3 * h)]
        q[h] = kinds[rng.integers(0, len(kinds), size=wl.n_tokens)]
    report_peaky("equal", run_case(wl, q, q, v, peaky=True))


def signs(wl, seed):
    """Vectors of 64 ones and minus ones: norms of 8 and products that are small whole numbers, so that similarities are either equal or differ by 1/32, in fp32 and
    in the oracle's arithmetic alike."""
    rng = np.random.default_rng(seed)
    return np.where(rng.integers(0, 2, size=(wl.heads, wl.n_tokens, 64)) > 0, 0x3f80, 0xbf80).astype(np.uint16)


@pytest.mark.parametrize("heads,frames", [(2, 3), (24, 23)], ids=["few", "many"])
@pytest.mark.parametrize("blk,ratio_q,ratio_kv", [((1, 3, 5), 0.5, 0.2), ((2, 4, 4), 0.3, 0.6), ((3, 4, 4), 0.6, 0.25), ((4, 4, 4), 0.5, 0.7), ((2, 5, 6), 0.1, 0.6),
                                                  ((2, 8, 8), 0.5, 0.7), ((1, 5, 13), 0.3, 0.5), ((4, 8, 8), 0.6, 0.2), ((4, 8, 9), 0.4, 0.6)],
                         ids=["15", "32", "48", "64", "60", "128", "65", "256", "288"])
def test_equal_similarities_go_by_position(blk, ratio_q, ratio_kv, heads, frames):
    """Exactly equal similarities: the best dst token is the first of them, and of the src tokens on the line between those that merge and the others those at the
    lowest positions merge.  The maps are the oracle's, token by token."""
    wl = synth.Workload("signs", frames, 2 * blk[1] + 3, 2 * blk[2] + 1, *blk, ratio_q, ratio_kv, n_camera=1, n_register=1, heads=heads, seed=1)
    q, k, v = (signs(wl, seed) for seed in (3, 4, 5))
    want = orc.global_attention(orc.Geometry.of(wl), ratio_q, ratio_kv, q, k, v, attend=False)
    assert (want.margin_sel_q == 0).any() and (want.margin_sel_k == 0).any() and (want.margin_best_q == 0).any()
    got = run(hb.HttmConfig.of(wl), [hb.bf16_from_bits(x, "cuda:0") for x in (q, k, v)])
    assert np.array_equal(got["assign_q"], want.assign_q) and np.array_equal(got["assign_k"], want.assign_k)
