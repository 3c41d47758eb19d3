"""Calls that follow one another on a stream without a wait between them: every kernel starts while the one before it is still
running (programmatic dependent launch), so a kernel that read too early would see the other call's intermediates.  Two inputs
alternate on one context; every output must be bit for bit what the input gives on its own."""
import pytest
import torch

from paper_2511_21317_b200 import binding as hb
from paper_2511_21317_b200 import synth

CASES = {   # the kernel families: warp per block, with filtering, with an anchored first frame; several passes; large blocks, with filtering
    "blocks_32": (dict(), 0.0),
    "blocks_32_filtered": (dict(), 0.05),
    "anchored": (dict(blk_frames=3), 0.0),
    "blocks_64": (dict(blk_frames=4), 0.0),
    "blocks_64_filtered": (dict(blk_frames=4), 0.05),
    "blocks_480": (dict(blk_frames=3, blk_h=10, blk_w=16), 0.0),
    "blocks_480_filtered": (dict(blk_frames=3, blk_h=10, blk_w=16), 0.05),
}


@pytest.mark.gpu
@pytest.mark.parametrize("name", sorted(CASES))
def test_alternating_inputs_without_waits(name):
    geometry, fraction = CASES[name]
    wl = synth.WORKLOADS["tiny"].replace(frames=7, grid_h=13, grid_w=18, **geometry)
    cfg = hb.HttmConfig.of(wl)
    if name == "anchored":
        cfg = hb.HttmConfig(**{**cfg.__dict__, "anchor_first_frame": 1})
    sets = []
    for seed in (1, 2):
        sets.append([hb.bf16_from_bits(x, "cuda:0") for x in synth.make_qkv(wl.replace(seed=seed))])
    with hb.Httm(cfg) as ctx:
        ctx.set_outlier_fraction(fraction)
        alone = []
        for qkv in sets:
            alone.append(ctx.global_attention(*qkv))
            torch.cuda.synchronize()
        assert not torch.equal(alone[0], alone[1])
        outs = [ctx.new_output() for _ in range(12)]
        for i, out in enumerate(outs):
            ctx.global_attention(*sets[i & 1], out)
        torch.cuda.synchronize()
        assert ctx.query(hb.Q_DEVICE_STATUS) == 0
        for i, out in enumerate(outs):
            assert torch.equal(out, alone[i & 1]), i


@pytest.mark.gpu
@pytest.mark.parametrize("name", ["blocks_32", "blocks_32_filtered", "blocks_64", "blocks_480_filtered"])
def test_inputs_written_right_before_the_call(name):
    """Merge, deviation and unmerge kernels read data of kernels further back while their predecessor still runs: the projection that
    writes Q, K and V in front of a call (it lets its successor start early, too) must be complete all the same."""
    geometry, fraction = CASES[name]
    wl = synth.WORKLOADS["tiny"].replace(frames=7, grid_h=13, grid_w=18, **geometry)
    n, dim = wl.n_tokens, wl.heads * 64
    gen = torch.Generator(device="cuda:0").manual_seed(3)
    xs = [torch.randn(n, dim, device="cuda:0", generator=gen).bfloat16() for _ in range(2)]
    w = (torch.randn(3 * dim, dim, device="cuda:0", generator=gen) / dim ** 0.5).bfloat16()
    qkv = torch.empty(n, 3 * dim, dtype=torch.bfloat16, device="cuda:0")
    views = [qkv[:, i * dim:(i + 1) * dim].view(n, wl.heads, 64).transpose(0, 1) for i in range(3)]
    with hb.Httm(hb.HttmConfig.of(wl)) as ctx:
        ctx.set_outlier_fraction(fraction)
        alone, merged = [], []
        for x in xs:
            ctx.linear(x, w, qkv)
            torch.cuda.synchronize()
            alone.append(ctx.global_attention(*views))
            torch.cuda.synchronize()
            merged.append(ctx.export(hb.X_K_MERGED))
        outs = [ctx.new_output() for _ in range(12)]
        for i, out in enumerate(outs):
            ctx.linear(xs[i & 1], w, qkv)
            ctx.global_attention(*views, out)
        torch.cuda.synchronize()
        assert ctx.query(hb.Q_DEVICE_STATUS) == 0
        for i, out in enumerate(outs):
            assert torch.equal(out, alone[i & 1]), i
        if name == "blocks_32":   # a stage on its own waits for whatever is in front of it (maps: those of the last call)
            for _ in range(4):
                ctx.linear(xs[0], w, qkv)
                ctx.linear(xs[1], w, qkv)
                ctx.launch_stage(hb.STAGE_MERGE_DIRECT, *views)
                torch.cuda.synchronize()
                assert (ctx.export(hb.X_K_MERGED) == merged[1]).all()
