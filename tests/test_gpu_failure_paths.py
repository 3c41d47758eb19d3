"""The error paths the library promises, provoked from the host (nothing here faults or hangs the device):
an allocation that fails (HTTM_ERR_NOMEM, everything taken so far is given back) and a bounded device-side wait
that runs out (the kernel returns, the status word is set, the host reports HTTM_ERR_TIMEOUT, the context stays
usable).  Needs a B200."""
import time

import numpy as np
import pytest
import torch

from paper_2511_21317_b200 import binding as hb
from paper_2511_21317_b200 import synth

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def test_failed_allocation_is_reported_and_nothing_leaks():
    wl = synth.WORKLOADS["tiny"]
    cfg = hb.HttmConfig.of(wl)
    with hb.Httm(cfg):                      # (loads the library's device code, so that the readings below are comparable)
        pass
    torch.cuda.synchronize()
    free0 = torch.cuda.mem_get_info()[0]
    try:
        for nth in (1, 2, 7, 15):           # the first allocation of httm_create, early ones, the last of the base workspace
            hb.fail_nth_allocation(nth)
            with pytest.raises(hb.HttmError) as e:
                hb.Httm(cfg)
            assert e.value.code == hb.ERR_NOMEM and "cudaMalloc" in str(e.value)
            assert torch.cuda.mem_get_info()[0] == free0, f"allocation {nth}: device memory was not given back"
        hb.fail_nth_allocation(0)
        with hb.Httm(cfg) as ctx:
            base = ctx.query(hb.Q_WORKSPACE_BYTES)
            free1 = torch.cuda.mem_get_info()[0]
            hb.fail_nth_allocation(4)       # inside the workspace of the outlier filter
            with pytest.raises(hb.HttmError) as e:
                ctx.set_outlier_fraction(0.1)
            assert e.value.code == hb.ERR_NOMEM
            assert ctx.query(hb.Q_WORKSPACE_BYTES) == base and torch.cuda.mem_get_info()[0] == free1
            ctx.set_outlier_fraction(0.1)   # the retry allocates everything and works
            q, k, v = (hb.bf16_from_bits(x, DEV) for x in synth.make_qkv(wl))
            out = ctx.global_attention(q, k, v)
            torch.cuda.synchronize()
            assert ctx.query(hb.Q_DEVICE_STATUS) == 0 and torch.isfinite(out.float()).all()
    finally:
        hb.fail_nth_allocation(0)


def test_an_expired_wait_is_reported_as_a_timeout_and_the_context_stays_usable():
    wl = synth.WORKLOADS["tiny"].replace(heads=2)
    q, k, v = (hb.bf16_from_bits(x, DEV) for x in synth.make_qkv(wl))
    with hb.Httm(hb.HttmConfig.of(wl)) as ctx:
        ref = ctx.global_attention(q, k, v).clone()
        torch.cuda.synchronize()
        assert ctx.query(hb.Q_DEVICE_STATUS) == 0
        t0 = time.perf_counter()
        ctx.expire_a_wait()                 # the kernel gives up after about two seconds and RETURNS
        torch.cuda.synchronize()
        waited = time.perf_counter() - t0
        assert 1.0 < waited < 10.0, waited
        with pytest.raises(hb.HttmError) as e:
            ctx.query(hb.Q_DEVICE_STATUS)
        assert e.value.code == hb.ERR_TIMEOUT
        with pytest.raises(hb.HttmError) as e:
            ctx.export(hb.X_ASSIGN_Q)
        assert e.value.code == hb.ERR_TIMEOUT
        again = ctx.global_attention(q, k, v)          # the device context and the library's context still work
        torch.cuda.synchronize()
        assert torch.equal(again, ref)
    with hb.Httm(hb.HttmConfig.of(wl)) as fresh:       # ... and so does a new one
        out = fresh.global_attention(q, k, v)
        torch.cuda.synchronize()
        assert fresh.query(hb.Q_DEVICE_STATUS) == 0 and torch.equal(out, ref)


# (frames, grid, blocks, ratio_q, ratio_kv, special tokens, heads, outlier fraction): query tiles are split over CTAs in all of them.
# The call's first kernel: match of small and of larger blocks, and reorder (special tokens, filter over sorted groups, large blocks)
SPLIT = {
    "unmerge_in_the_epilogue": (4, (37, 37), (2, 4, 4), 0.9, 0.0, 5, 2, 0.0),
    "per_head_lengths": (8, (37, 37), (2, 4, 4), 0.8, 0.2, 5, 2, 0.03),
    "blocks_64": (11, (37, 37), (4, 4, 4), 0.9, 0.0, 5, 1, 0.0),
    "over_reordered_copies": (4, (37, 37), (2, 4, 4), 0.9, 0.0, 40, 2, 0.0),
    "sorted_groups": (8, (37, 37), (4, 4, 4), 0.8, 0.2, 5, 2, 0.03),
    "large_blocks": (8, (1, 1024), (8, 1, 128), 0.9, 0.2, 5, 2, 0.0),
}


@pytest.mark.parametrize("name", sorted(SPLIT))
def test_parts_that_an_earlier_call_left_unfinished(name):
    """An attention kernel that gives up leaves arrivals of split query tiles counted; later calls and stages give the same bits all the same."""
    frames, grid, blk, rq, rkv, specials, heads, fraction = SPLIT[name]
    wl = synth.Workload(name, frames, *grid, *blk, rq, rkv, n_camera=1, n_register=specials - 1, heads=heads, seed=3)
    q, k, v = (hb.bf16_from_bits(x, DEV) for x in synth.make_qkv(wl))
    reorders = name in ("over_reordered_copies", "sorted_groups", "large_blocks")
    with hb.Httm(hb.HttmConfig.of(wl)) as ctx:
        ctx.set_outlier_fraction(fraction)
        ref = ctx.global_attention(q, k, v).clone()
        merged = ctx.export(hb.X_O_MERGED)
        assert ctx.query(hb.Q_DEVICE_STATUS) == 0

        def other_call():          # rows that are not written hold another call's values, not the right ones
            ctx.global_attention(q, k, -v)
            ctx.export(hb.X_O_MERGED)
            ctx.leave_parts_unfinished()

        for _ in range(2):
            out = torch.zeros_like(ref)
            other_call()
            ctx.global_attention(q, k, v, out)
            torch.cuda.synchronize()
            assert torch.equal(out, ref)
        # the attention on its own, as a stage and behind an export
        other_call()
        if reorders:
            ctx.launch_stage(hb.STAGE_REORDER, q, k, v)
        ctx.launch_stage(hb.STAGE_MERGE if reorders else hb.STAGE_MERGE_DIRECT, q, k, v)
        out = torch.zeros_like(ref)
        ctx.launch_stage(hb.STAGE_ATTENTION)
        ctx.launch_stage(hb.STAGE_UNMERGE, out=out)
        torch.cuda.synchronize()
        assert torch.equal(out, ref)
        if not fraction:           # (rows past a head's merged length are not defined)
            other_call()
            ctx.global_attention(q, k, v)
            ctx.leave_parts_unfinished()
            assert np.array_equal(ctx.export(hb.X_O_MERGED), merged)
        assert ctx.query(hb.Q_DEVICE_STATUS) == 0
