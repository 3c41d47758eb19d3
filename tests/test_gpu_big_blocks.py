"""Parity of the large-block path (merging blocks of 257 .. 4096 tokens: the paper's runs of 128 tokens over 30
frames, Sec. 3.3 / 4.1) with the CPU oracle.  All tests here need a B200."""
import dataclasses

import numpy as np
import pytest
import torch

from oracle import httm_oracle as orc
from paper_2511_21317_b200 import binding as hb
from paper_2511_21317_b200 import synth
from tests import parity
from tests.test_gpu_parity import exports

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def run_big(wl, q=None, k=None, v=None, sample=None, peaky=False):
    if q is None:
        q, k, v = synth.make_qkv(wl)
    g = orc.Geometry.of(wl)
    with hb.Httm(hb.HttmConfig.of(wl)) as ctx:
        assert ctx.query(hb.Q_MAX_BLOCK_TOKENS) > 256
        assert ctx.m_q == orc.merged_len(g, wl.ratio_q) and ctx.m_k == orc.merged_len(g, wl.ratio_kv)
        dq, dk, dv = (hb.bf16_from_bits(x, DEV) for x in (q, k, v))
        before = ctx.launch_count()
        out = ctx.global_attention(dq, dk, dv)
        torch.cuda.synchronize()
        assert ctx.launch_count() - before == 6          # reorder, scores, select, merge, attention, unmerge
        assert ctx.query(hb.Q_DEVICE_STATUS) == 0
        ex = exports(ctx)
        stats = parity.full_check(g, wl.ratio_q, wl.ratio_kv, q, k, v, ex, hb.bits_from_bf16(out), sample, wl.name, peaky)
        out2 = ctx.global_attention(dq, dk, dv)
        torch.cuda.synchronize()
        assert torch.equal(out, out2)
        ex2 = exports(ctx)
        for name in ex:
            assert np.array_equal(ex[name], ex2[name]), f"{name} differs between two identical calls"
        # the stages one by one give the same result
        out3 = ctx.new_output()
        for st in (hb.STAGE_REORDER, hb.STAGE_BIG_SCORES, hb.STAGE_BIG_SELECT, hb.STAGE_MERGE, hb.STAGE_ATTENTION, hb.STAGE_UNMERGE):
            ctx.launch_stage(st, dq, dk, dv, out3)
        torch.cuda.synchronize()
        assert torch.equal(out, out3)
        for st in (hb.STAGE_MATCH, hb.STAGE_MATCH_DIRECT, hb.STAGE_MERGE_DIRECT):
            with pytest.raises(hb.HttmError) as e:
                ctx.launch_stage(st, dq, dk, dv, out3)
            assert e.value.code == hb.ERR_UNSUPPORTED
    return stats


GEOMS = [
    # name, frames, grid_h, grid_w, blk, ratio_q, ratio_kv, n_camera, n_register, heads
    ("runs_ragged", 4, 1, 230, (4, 1, 100), 0.9, 0.7, 1, 0, 2),            # blocks of 400, 400, 120 tokens
    ("windows_512", 5, 17, 19, (4, 8, 16), 0.7, 0.5, 1, 4, 2),             # 2-D windows, clipped in every direction
    ("just_above_256", 3, 10, 30, (3, 9, 10), 0.6, 0.8, 1, 4, 2),          # 270-token blocks
    ("runs_3840", 30, 1, 300, (30, 1, 128), 0.9, 0.7, 1, 4, 2),            # the paper's block: 3840, 3840, 1320 tokens
    ("max_4096", 32, 1, 140, (32, 1, 128), 0.75, 0.9, 1, 0, 1),            # 4096-token block + a ragged one
    ("ratio_zero_q", 4, 1, 300, (4, 1, 128), 0.0, 0.7, 1, 4, 2),
    ("ratio_099", 4, 1, 300, (4, 1, 128), 0.99, 0.99, 1, 4, 2),
    ("odd_dst_counts", 7, 1, 211, (7, 1, 97), 0.83, 0.41, 0, 0, 3),        # n = 679, 679, 119: n_dst not a multiple of anything
]


@pytest.mark.parametrize("case", GEOMS, ids=[c[0] for c in GEOMS])
def test_large_block_geometries(case):
    name, S, h, w, blk, rq, rkv, ncam, nreg, H = case
    wl = synth.Workload(name, S, h, w, blk[0], blk[1], blk[2], rq, rkv, n_camera=ncam, n_register=nreg, heads=H, seed=5)
    run_big(wl, peaky=True)


def test_large_blocks_random_uncorrelated_inputs():
    wl = synth.Workload("gauss_big", 8, 1, 200, 8, 1, 128, 0.8, 0.6, heads=3)
    rng = np.random.default_rng(11)
    q, k, v = (synth.f32_to_bf16_bits(rng.standard_normal((wl.heads, wl.n_tokens, 64)).astype(np.float32)) for _ in range(3))
    run_big(wl, q, k, v, peaky=True)


def test_large_blocks_ties_and_zero_vectors():
    """Identical tokens in a block: every cosine ties, all src go to the first dst (one group of hundreds of tokens)."""
    wl = synth.Workload("ties_big", 4, 1, 150, 4, 1, 100, 0.5, 0.5, heads=2, n_camera=1, n_register=1)
    x = synth.make_identical_block_tokens(wl, seed=4)
    q, k, v = synth.make_qkv(wl)
    z = q.copy()
    z[:, 10:400, :] = 0
    run_big(wl, x, k, v, peaky=True)
    run_big(wl, q, x, v, peaky=True)
    run_big(wl, z, z, v, peaky=True)


def test_paper_block_regime_full_size_sampled():
    """Runs of 128 tokens x 30 frames on 60 frames of 37 x 37 patches, 90 % / 70 % merged (Sec. 4.1), all 16 heads (the
    configuration the benchmark times): maps and merged tensors on all tokens, attention output on sampled tokens."""
    wl = synth.WORKLOADS["paper_1d"]
    rng = np.random.default_rng(2)
    toks = np.unique(np.concatenate([rng.integers(0, wl.n_tokens, 24), [0, 4, 5, wl.n_tokens - 1]]))
    stats = run_big(wl, sample=toks)
    assert stats["out_err"] <= parity.OUT_TOL and stats["peaky_needed"] == 0


@pytest.mark.parametrize("n", [511, 512, 513, 1023, 1025, 2047, 2048, 2049, 4095])
def test_block_sizes_at_the_cta_size_limits(n):
    """One block of n tokens per head: the sorted-group kernels take 4 tokens per thread of a 128 .. 512-thread CTA, 8 above
    2048 tokens; many groups (two counting passes) for the queries, at most 64 (one pass) for the keys."""
    wl = synth.Workload(f"one_block_{n}", 1, 1, n, 1, 1, n, 0.7, 1.0 - 60.0 / n, n_camera=0, n_register=2, heads=2, seed=n)
    run_big(wl, peaky=True)
    if n in (513, 2049):
        from tests.test_gpu_outlier import run_filtered
        run_filtered(wl, 0.1, peaky=True, launches=12)


@pytest.mark.parametrize("n", [257, 260, 508, 516, 1028, 3844, 4096])
def test_dst_tokens_at_the_chunk_limits(n):
    """One block of n tokens per head, a quarter of them dst tokens: 65, 127 and 129 of them (chunks of 128, halves of 64, parts of 32),
    257, 961 and 1024; even and odd numbers of token tiles, the last with one row or full."""
    wl = synth.Workload(f"dst_limit_{n}", 1, 1, n, 1, 1, n, 0.7, 0.5, n_camera=0, n_register=1, heads=3, seed=n)
    run_big(wl, peaky=True)


@pytest.mark.parametrize("bad", [float("inf"), float("nan"), 2.0 ** 70], ids=["infinite", "not_a_number", "overflow"])
def test_a_dst_token_without_a_similarity_is_nobodys_best(bad):
    """Dst tokens that are infinite, not numbers or of a squared norm beyond fp32: the other tokens go to the best of the other dst tokens (all
    similarities of this scene are positive), to within the rounding of the similarities (1e-5)."""
    n, heads = 1100, 2
    wl = synth.Workload("spoilt", 1, 1, n, 1, 1, n, 0.75, 0.75, n_camera=0, n_register=0, heads=heads, seed=3)
    gen = np.random.default_rng(7)
    x = (0.25 + gen.random((heads, n, 64))).astype(np.float32)
    nd = n // 4
    dst = np.arange(3, n, 4)
    spoilt = dst[[0, 31, 32, 100, 274]]
    x[:, spoilt] *= bad
    t = torch.from_numpy(x).bfloat16().to(DEV)
    good = torch.from_numpy((0.25 + gen.random(x.shape)).astype(np.float32)).bfloat16().to(DEV)
    with hb.Httm(hb.HttmConfig.of(wl)) as ctx:
        ctx.global_attention(t, t, good)
        torch.cuda.synchronize()
        assert ctx.query(hb.Q_DEVICE_STATUS) == 0
        maps = ctx.export(hb.X_ASSIGN_Q), ctx.export(hb.X_ASSIGN_K)
    rows = t.double().cpu().numpy()
    src, fine = np.setdiff1d(np.arange(n), dst), np.setdiff1d(dst, spoilt)
    assert len(src) == int(0.75 * n) and len(dst) == nd
    for h in range(heads):
        with np.errstate(all="ignore"):
            unit = rows[h] / np.linalg.norm(rows[h], axis=1, keepdims=True)
        sim = unit[src] @ unit[fine].T
        for m in maps:
            assert np.isin(m[h][src], fine).all() and (m[h][dst] == dst).all()
            mine = (unit[src] * unit[m[h][src]]).sum(1)
            assert (sim.max(1) - mine <= 1e-5).all(), (h, (sim.max(1) - mine).max())


def test_norms_far_from_one_change_no_map():
    """Every token multiplied by a power of two of its own, 2^-30 .. 2^60 (squared norms stay inside fp32, norms above the clamp): products,
    norms and weights scale exactly, so the maps are the same."""
    n, heads = 1500, 2
    wl = synth.Workload("scaled", 1, 1, n, 1, 1, n, 0.7, 0.4, n_camera=0, n_register=1, heads=heads, seed=4)
    q, k, v = synth.make_qkv(wl)
    gen = np.random.default_rng(9)
    maps = []
    for scaled in (False, True):
        with hb.Httm(hb.HttmConfig.of(wl)) as ctx:
            dq, dk, dv = (hb.bf16_from_bits(x, DEV) for x in (q, k, v))
            if scaled:
                dq, dk = (t * torch.exp2(torch.from_numpy(gen.integers(-30, 61, t.shape[:2])).float()).to(DEV).bfloat16()[..., None] for t in (dq, dk))
            ctx.global_attention(dq, dk, dv)
            torch.cuda.synchronize()
            assert ctx.query(hb.Q_DEVICE_STATUS) == 0
            maps.append((ctx.export(hb.X_ASSIGN_Q), ctx.export(hb.X_ASSIGN_K)))
    for a, b in zip(*maps):
        assert np.array_equal(a, b)


def test_sums_of_many_members_with_one_far_larger_member():
    """2 048 tokens in one block, multiples of one vector (every cosine a tie: nearly all of them merge into the first dst token), one of
    them 2^17 times the others.  In fp32 every small member added to a running sum of that size is rounded in the same direction, so a
    sum in position order is off by up to half a unit in the last place per member.  The bound is that of four running sums of every fourth
    member each, (n / 4 + 2) roundings of at most 2^-24 of the sum of magnitudes."""
    n, heads = 2048, 4
    wl = synth.Workload("large_member", 1, 1, n, 1, 1, n, 0.99, 0.99, n_camera=0, n_register=1, heads=heads, seed=0)
    gen = np.random.default_rng(5)
    u = (1.0 + gen.integers(0, 128, (heads, 1, 64)) / 128.0) * gen.choice([-1.0, 1.0], (heads, 1, 64))
    x = np.repeat(u, n + 1, axis=1)
    x[:, 1] *= 2.0 ** 17
    t = torch.from_numpy(x).bfloat16().to(DEV)
    assert (t.double().cpu().numpy() == x).all()
    with hb.Httm(hb.HttmConfig.of(wl)) as ctx:
        ctx.set_outlier_fraction(1e-4)
        ctx.global_attention(t, t, t)
        torch.cuda.synchronize()
        assert ctx.query(hb.Q_DEVICE_STATUS) == 0
        aq, ak = ctx.export(hb.X_ASSIGN_Q_INITIAL), ctx.export(hb.X_ASSIGN_K)
        eps = ctx.export(hb.X_DEVIATION).astype(np.float64)
        k_m, v_m = (parity.bits_to_f64(ctx.export(w)) for w in (hb.X_K_MERGED, hb.X_V_MERGED))
    roundings = (n / 4 + 2) * 2.0 ** -24
    for h in range(heads):
        members = np.flatnonzero(aq[h] == aq[h][1])
        assert len(members) > 0.98 * n and members[0] == 1
        mean, size = x[h][members].mean(0), np.abs(x[h][members]).mean(0)
        want = np.linalg.norm(x[h][members] - mean, axis=1)
        bound = np.linalg.norm(roundings * size) + (64 + 4) * 2.0 ** -24 * want      # the mean, then differences, 64 squares and the root
        assert (np.abs(eps[h][members] - want) <= bound).all(), (h, np.abs(eps[h][members] - want).max(), bound.max())
        kept = np.flatnonzero(ak[h] == np.arange(n + 1))
        members = np.flatnonzero(ak[h] == ak[h][1])
        mean, size = x[h][members].mean(0), np.abs(x[h][members]).mean(0)
        row = np.flatnonzero(kept == ak[h][1])[0]
        for got in (k_m[h][row], v_m[h][row]):   # within half a bf16 step of the mean, up to the same bound
            step = 2.0 ** (np.floor(np.log2(np.abs(mean))) - 7)
            assert (np.abs(got - mean) <= step / 2 + roundings * size).all(), (h, (np.abs(got - mean) / step).max())


def similarities(x, src, dst):
    """What a similarity is where fp32 cannot hold a square (x [n][64], values of bf16 in float64): weights 1 / max(norm, 1e-12) from the squared
    norm in fp32 (0 where it overflows), the product of a src token with a weighted dst token, weighted by the src token's own weight.  Returns the weighted
    products [src][dst] and the weights of the src tokens."""
    with np.errstate(all="ignore"):
        w = np.minimum(1.0 / np.sqrt((x * x).sum(1).astype(np.float32).astype(np.float64)), 1e12)
        return x[src] @ (x[dst] * w[dst, None]).T, w[src]


@pytest.mark.parametrize("dst_scale", [0, 27, -74])
@pytest.mark.parametrize("src_scale", [-74, 68, 98, 120])
def test_products_that_fp32_does_not_hold(src_scale, dst_scale):
    """Every third src token times 2^src_scale, every dst token times 2^dst_scale (rows of norms around 5): their products leave fp32's range, but the
    products with dst tokens of norm one do not.  A src token goes to the dst token of the largest weighted product; one whose squared
    norm overflows has weight 0 and similarity 0: it merges behind the others, such tokens in position order."""
    n, heads = 900, 2
    r = int(0.7 * n)
    wl = synth.Workload("range", 1, 1, n, 1, 1, n, 0.7, 0.7, n_camera=0, n_register=0, heads=heads, seed=3)
    gen = np.random.default_rng(21)
    x = (0.25 + gen.random((heads, n, 64))).astype(np.float32)
    nd = n // 4
    dst = np.array([j for j in range(n) if (j + 1) * nd // n > j * nd // n])
    src = np.setdiff1d(np.arange(n), dst)
    far = src[::3]
    assert len(src) - len(far) < r < len(src)   # some of the scaled tokens merge, some do not
    x[:, far] *= 2.0 ** src_scale
    x[:, dst] *= 2.0 ** dst_scale
    t = torch.from_numpy(x).bfloat16().to(DEV)
    good = torch.from_numpy((0.25 + gen.random(x.shape)).astype(np.float32)).bfloat16().to(DEV)
    with hb.Httm(hb.HttmConfig.of(wl)) as ctx:
        ctx.global_attention(t, t, good)
        torch.cuda.synchronize()
        assert ctx.query(hb.Q_DEVICE_STATUS) == 0
        maps = ctx.export(hb.X_ASSIGN_Q), ctx.export(hb.X_ASSIGN_K)
    rows = t.double().cpu().numpy()
    for h in range(heads):
        prod, w = similarities(rows[h], src, dst)
        best, key = prod.max(1), prod.max(1) * w
        for m in maps:
            to = m[h][src]
            merged = to != src
            assert merged.sum() == r and (m[h][dst] == dst).all() and np.isin(to[merged], dst).all()
            mine = prod[np.flatnonzero(merged), np.searchsorted(dst, to[merged])]
            assert (mine >= best[merged] * (1 - 1e-5)).all(), (h, (1 - mine / best[merged]).max())
            assert key[merged].min() >= key[~merged].max() - 1e-5 * abs(key).max()
            if src_scale > 64:   # weight 0: equal similarities, the lowest positions merge
                tied = np.flatnonzero(w == 0)
                assert len(tied) == len(far) and (np.diff(merged[tied].astype(int)) <= 0).all()


@pytest.mark.parametrize("dst_scale", [0, 27])
def test_infinite_src_tokens_merge_first(dst_scale):
    """An infinite src token: its weight is 0, its similarity 0 x infinity, whose key orders above all numbers, as in the kernels of smaller blocks.
    All its products are infinite here: the lowest dst token."""
    n, heads = 900, 2
    wl = synth.Workload("infinite", 1, 1, n, 1, 1, n, 0.5, 0.5, n_camera=0, n_register=0, heads=heads, seed=3)
    gen = np.random.default_rng(22)
    x = (0.25 + gen.random((heads, n, 64))).astype(np.float32)
    nd = n // 4
    dst = np.array([j for j in range(n) if (j + 1) * nd // n > j * nd // n])
    src = np.setdiff1d(np.arange(n), dst)
    far, near = src[5::7], np.setdiff1d(src, src[5::7])
    x[:, dst] *= 2.0 ** dst_scale
    x[:, far] = np.inf
    t = torch.from_numpy(x).bfloat16().to(DEV)
    good = torch.from_numpy((0.25 + gen.random(x.shape)).astype(np.float32)).bfloat16().to(DEV)
    with hb.Httm(hb.HttmConfig.of(wl)) as ctx:
        ctx.global_attention(t, t, good)
        torch.cuda.synchronize()
        assert ctx.query(hb.Q_DEVICE_STATUS) == 0
        maps = ctx.export(hb.X_ASSIGN_Q), ctx.export(hb.X_ASSIGN_K)
    rows = t.double().cpu().numpy()
    for h in range(heads):
        prod, w = similarities(rows[h], near, dst)
        key = prod.max(1) * w
        for m in maps:
            assert (m[h][far] == dst[0]).all()
            merged = m[h][near] != near
            assert merged.sum() == n // 2 - len(far)
            assert key[merged].min() >= key[~merged].max() - 1e-5


@pytest.mark.parametrize("column", [0, 5])
@pytest.mark.parametrize("bad", [float("inf"), float("nan")], ids=["infinite", "not_a_number"])
@pytest.mark.parametrize("first", [16, 72, 200], ids=["same_part", "other_half", "later_chunk"])
def test_equal_best_dst_tokens_beside_one_without_a_similarity(first, bad, column):
    """Src tokens equal to two dst tokens among eight neighbours, and a dst token without a similarity at the first one's place among
    eight others: they go to the first of the two."""
    n, heads = 1100, 2
    wl = synth.Workload("spoilt_ties", 1, 1, n, 1, 1, n, 0.75, 0.75, n_camera=0, n_register=0, heads=heads, seed=3)
    gen = np.random.default_rng(23)
    x = gen.standard_normal((heads, n, 64)).astype(np.float32)
    nd = n // 4
    dst = np.array([j for j in range(n) if (j + 1) * nd // n > j * nd // n])
    src = np.setdiff1d(np.arange(n), dst)
    low, high = dst[first + column], dst[first + 7]
    same = src[::5]
    x[:, high] = x[:, low]
    x[:, same] = x[:, low][:, None]
    x[:, dst[column + (64 if first > 64 else 0)]] = bad
    t = torch.from_numpy(x).bfloat16().to(DEV)
    good = torch.from_numpy(gen.standard_normal(x.shape).astype(np.float32)).bfloat16().to(DEV)
    with hb.Httm(hb.HttmConfig.of(wl)) as ctx:
        ctx.global_attention(t, t, good)
        torch.cuda.synchronize()
        assert ctx.query(hb.Q_DEVICE_STATUS) == 0
        maps = ctx.export(hb.X_ASSIGN_Q), ctx.export(hb.X_ASSIGN_K)
    for m in maps:
        assert (m[:, same] == low).all()


@pytest.mark.parametrize("ratio_q,ratio_kv,anchor", [(0.9, 0.7, 0), (0.0, 0.5, 0), (0.6, 0.7, 1)], ids=["five_stages", "queries_not_merged", "anchored"])
def test_several_blocks_per_cta_agree_with_one(ratio_q, ratio_kv, anchor):
    """The score kernel's CTAs take blocks from a counter and carry the state of their rings and buffers from one to the next: 18 blocks (ten of 4096 tokens, of up to
    1024 dst tokens; two of 96, five of 128, one of 3) x 16 heads x 2 tensors are four per CTA.  One head at a time every CTA takes at most one: the same maps."""
    wl = synth.Workload("several", 65, 1, 643, 32, 1, 128, ratio_q, ratio_kv, n_camera=1, n_register=0, heads=16, seed=3)
    gen = torch.Generator(device=DEV).manual_seed(5)
    q, k, v = (torch.randn(wl.heads, wl.n_tokens, 64, generator=gen, device=DEV).bfloat16() for _ in range(3))

    def maps(*tensors):
        ctx.global_attention(*tensors)
        torch.cuda.synchronize()
        assert ctx.query(hb.Q_DEVICE_STATUS) == 0
        return ctx.export(hb.X_ASSIGN_Q), ctx.export(hb.X_ASSIGN_K)

    with hb.Httm(dataclasses.replace(hb.HttmConfig.of(wl), anchor_first_frame=anchor)) as ctx:
        together = maps(q, k, v)
    with hb.Httm(dataclasses.replace(hb.HttmConfig.of(wl.replace(heads=1)), anchor_first_frame=anchor)) as ctx:
        for h in range(wl.heads):
            alone = maps(q[h:h + 1], k[h:h + 1], v[h:h + 1])
            for m, one in zip(together, alone):
                assert np.array_equal(m[h], one[0]), h


@pytest.mark.parametrize("heads,frames,width,run", [(1, 11, 700, 128), (2, 9, 300, 64), (1, 5, 131, 131), (3, 30, 257, 96), (5, 7, 520, 128)])
def test_blocks_shared_out_to_several_ctas(heads, frames, width, run):
    """Few blocks: their src tokens go to several score CTAs, their groups to several merge CTAs (one to four, with odd numbers of tiles), and the
    same heads among many others to one score CTA and one or two merge CTAs: the same maps, ranks and merged tensors, bit for bit."""
    wl = synth.Workload("shares", frames, 1, width, frames, 1, run, 0.8, 0.6, n_camera=1, n_register=2, heads=heads, seed=11)
    many = wl.replace(heads=148)
    reps = -(-148 // heads)
    q, k, v = (np.tile(x, (reps, 1, 1))[:148] for x in synth.make_qkv(wl))
    items = {"assign_q": hb.X_ASSIGN_Q, "assign_k": hb.X_ASSIGN_K, "rank_q": hb.X_RANK_Q, "q_m": hb.X_Q_MERGED, "k_m": hb.X_K_MERGED, "v_m": hb.X_V_MERGED}
    got = {}
    for name, w, n in (("few", wl, heads), ("many", many, 148)):
        with hb.Httm(hb.HttmConfig.of(w)) as ctx:
            ctx.global_attention(*(hb.bf16_from_bits(x[:n], DEV) for x in (q, k, v)))
            torch.cuda.synchronize()
            assert ctx.query(hb.Q_DEVICE_STATUS) == 0
            got[name] = {i: ctx.export(x) for i, x in items.items()}
    for i in items:
        assert np.array_equal(got["few"][i], got["many"][i][:heads]), i
        assert np.array_equal(got["few"][i][0], got["many"][i][heads * (reps - 1)]), i


@pytest.mark.parametrize("heads,frames,width,run", [(1, 11, 700, 128), (2, 9, 300, 64), (1, 5, 131, 131), (3, 30, 257, 96), (5, 7, 520, 128)])
@pytest.mark.parametrize("fraction", [0.0, 0.1])
def test_heads_among_others_that_leave_one_cta_per_block(heads, frames, width, run, fraction):
    """So many other heads that every block has one CTA in all kernels, without outlier filtering and with it.  The threshold of the filter depends on all heads, so
    with it the deviations, which are of the map before, and what K's map gives are compared."""
    wl = synth.Workload("shares", frames, 1, width, frames, 1, run, 0.8, 0.6, n_camera=1, n_register=2, heads=heads, seed=11)
    blocks = -(-width // run)
    reps = -(-450 // (heads * blocks)) + 1   # (blocks of all heads; 888 CTAs of 256 threads that fold deviations fit at once, fewer of the others)
    n_many = heads * (reps - 1) + 1
    many = tuple(hb.bf16_from_bits(np.tile(t, (reps, 1, 1))[:n_many], DEV) for t in synth.make_qkv(wl))
    items = {"assign_k": hb.X_ASSIGN_K, "k_m": hb.X_K_MERGED, "v_m": hb.X_V_MERGED}
    items.update({"eps": hb.X_DEVIATION, "assign_q0": hb.X_ASSIGN_Q_INITIAL} if fraction else {"assign_q": hb.X_ASSIGN_Q, "rank_q": hb.X_RANK_Q, "q_m": hb.X_Q_MERGED})
    got = {}
    for name, n in (("few", heads), ("many", n_many)):
        with hb.Httm(hb.HttmConfig.of(wl.replace(heads=n))) as ctx:
            if fraction:
                ctx.set_outlier_fraction(fraction)
            ctx.global_attention(*(t[:n] for t in many))
            torch.cuda.synchronize()
            assert ctx.query(hb.Q_DEVICE_STATUS) == 0
            got[name] = {i: ctx.export(what) for i, what in items.items()}
    for i in items:
        assert np.array_equal(got["few"][i], got["many"][i][:heads]), i
        assert np.array_equal(got["few"][i][0], got["many"][i][heads * (reps - 1)]), i
    assert not fraction or (got["few"]["eps"] > 0).any()
