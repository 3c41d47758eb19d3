"""Tokens so large that their squared norm overflows in fp32 (or that are infinite): the similarity of two of them is not a number.  Such a
similarity is never the best one: the token goes to the best of the other dst tokens, in every match kernel.  Reference: the rule written
out in numpy with fp32's overflow."""
import numpy as np
import pytest
import torch

from paper_2511_21317_b200 import binding as hb
from paper_2511_21317_b200 import synth

pytestmark = pytest.mark.gpu


def map_of_block(x, ratio):
    """Map of one block of tokens x [n][64] (float32 holding bf16 values)."""
    n = len(x)
    r = min(int(np.floor(ratio * n + 1e-9)), n - 1)
    nd = min(-(-n // 4), n - r)
    dst = np.array([j for j in range(n) if (j + 1) * nd // n > j * nd // n])
    src = np.setdiff1d(np.arange(n), dst)
    with np.errstate(all="ignore"):
        x64 = x.astype(np.float64)
        square = (x64 * x64).sum(1).astype(np.float32)                 # inf where fp32 overflows
        inv = np.minimum(np.float32(1) / np.sqrt(square), np.float32(1e12))
        dot = (x64[src] @ x64[dst].T).astype(np.float32)
        sim = dot * inv[dst]
        sim = np.where(np.isnan(sim), np.float32(-np.inf), sim)
    best = sim.argmax(1)                                                # ties: the lowest dst
    assert r == len(src)                                                # every src token merges: the selection plays no part
    out = np.arange(n)
    out[src] = dst[best]
    return out


@pytest.mark.parametrize("every", [2, 1], ids=["every_other_dst", "every_dst"])
@pytest.mark.parametrize("big", [2.0 ** 70, float("inf")], ids=["overflow", "infinite"])
@pytest.mark.parametrize("blk", [(2, 4, 4), (4, 4, 4), (2, 8, 8), (4, 8, 8)], ids=["32", "64", "128", "256"])
def test_a_similarity_that_is_not_a_number_never_wins(blk, big, every):
    n = blk[0] * blk[1] * blk[2]
    wl = synth.Workload("nan", blk[0], blk[1] * 2, blk[2], *blk, 0.75, 0.75, n_camera=0, n_register=0, heads=3, seed=1)
    gen = np.random.default_rng(n)
    x = (0.25 + gen.random((wl.heads, wl.n_tokens, 64))).astype(np.float32)      # positive: every dot product is
    bf = lambda a: torch.from_numpy(a).bfloat16()
    probe = hb.Httm(hb.HttmConfig.of(wl))
    pi, start = probe.export(hb.X_PI), probe.export(hb.X_BLOCK_START)
    probe.close()
    nd = n // 4
    dst = np.array([j for j in range(n) if (j + 1) * nd // n > j * nd // n])
    src = np.setdiff1d(np.arange(n), dst)
    huge = np.concatenate([dst[::every], src[::3]])                               # dst tokens, and a third of the others
    for b in range(2):
        x[:, pi[start[b] + huge]] *= big
    t = bf(x).cuda()
    small = bf((0.25 + gen.random(x.shape)).astype(np.float32)).cuda()
    with hb.Httm(hb.HttmConfig.of(wl)) as ctx:
        ctx.global_attention(t, t, small)
        torch.cuda.synchronize()
        assert ctx.query(hb.Q_DEVICE_STATUS) == 0
        maps = ctx.export(hb.X_ASSIGN_Q), ctx.export(hb.X_ASSIGN_K)
    rows = bf(x).float().numpy()
    for h in range(wl.heads):
        for b in range(2):
            want = start[b] + map_of_block(rows[h][pi[start[b]:start[b + 1]]], 0.75)
            for m in maps:
                assert np.array_equal(m[h, start[b]:start[b + 1]], want), (h, b)
