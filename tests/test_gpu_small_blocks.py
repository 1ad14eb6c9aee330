"""64-token blocks: the kernel with one query block per CTA, work items of two and four of them, ragged ends, every mode."""
import numpy as np
import pytest
import torch

from paper_2607_24027_b200 import synth
from tests import helpers as hp
from tests.test_gpu_parity import _check_all_heads, _lib, _small_problem  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


# 148 SMs: up to 148 query blocks over all heads run as one block per CTA, up to 296 as items of two, more as items of
# four; a last item that lacks one, two or three of its blocks, and last blocks of 1, 63 and 64 tokens
@pytest.mark.parametrize("H,N,d", [(1, 64, 64), (2, 65, 128), (2, 64 * 37, 64), (20, 64 * 9 + 63, 128), (40, 64 * 8, 64),
                                   (40, 64 * 8 + 1, 128), (36, 64 * 9 + 63, 64), (30, 64 * 11, 128)])
@pytest.mark.parametrize("mode", ["sol", "exact_only", "dense"])
def test_item_shapes(H, N, d, mode):
    from paper_2607_24027_b200 import binding as sb
    bits = _small_problem(N + d, 1, H, N, d)
    if mode == "dense":
        q, k, v = (hp.to_dev(x) for x in bits)
        out, counts, _, _ = hp.run_gpu(q, k, v, 64, 0.0, mode=sb.SOL_MODE_DENSE)
        ref = torch.nn.functional.scaled_dot_product_attention(q.double(), k.double(), v.double())
        assert float((out.double() - ref).abs().max()) <= hp.MAX_ABS
        assert bool((counts == -(-N // 64)).all())
        return
    heads = sorted({0, H // 2, H - 1})                            # the oracle is slow: three heads of the same call
    out, counts, mask, _ = hp.run_gpu(*(hp.to_dev(x) for x in bits), 64, 0.5,
                                      mode=sb.SOL_MODE_SOL if mode == "sol" else sb.SOL_MODE_EXACT_ONLY)
    assert np.array_equal(counts.cpu().numpy(), mask.sum(axis=-1))
    o = hp.dev_to_f64(out)
    for h in heads:
        hp.check_head(*(synth.widen(b[0, h], np.float64) for b in bits), o[0, h], mask[0, h], counts[0, h].cpu().numpy(),
                      64, 0.5, mode=mode)


def test_a_neighbours_block_leaves_no_trace():
    """Four query blocks share a work item and its tiles, not their results: a key block whose values are not finite
    reaches only the query blocks that routed it, and a block that routes nothing is zero."""
    from paper_2607_24027_b200 import binding as sb
    H, N = 40, 64 * 12
    bits = _small_problem(5, 1, H, N, 64)
    q, k, v = (hp.to_dev(x) for x in bits)
    clean, counts, mask, ws = hp.run_gpu(q, k, v, 64, 1.0, mode=sb.SOL_MODE_EXACT_ONLY)
    v[:, :, 64 * 5:64 * 6] = float("inf")
    out, counts2, mask2, _ = hp.run_gpu(q, k, v, 64, 1.0, mode=sb.SOL_MODE_EXACT_ONLY, ws=ws)
    assert np.array_equal(mask, mask2)
    hit = torch.from_numpy(np.repeat(mask[0, :, :, 5], 64, axis=1)).cuda()      # [H, N]
    assert 0 < int(hit.sum()) < hit.numel()
    assert torch.equal(out[0][~hit].view(torch.int16), clean[0][~hit].view(torch.int16))
    assert not bool(torch.isfinite(out[0][hit]).any())
    none = torch.from_numpy(np.repeat(counts.cpu().numpy()[0] == 0, 64, axis=1)).cuda()
    assert bool((out[0][none] == 0).all())
    # more records without a single tile than the ring holds
    out, counts, _, _ = hp.run_gpu(q, k, v, 64, float("inf"), mode=sb.SOL_MODE_EXACT_ONLY, ws=ws)
    assert bool((out == 0).all()) and int(counts.sum()) == 0


def _many_blocks(B, H, N, d, seed):
    """More query blocks than SMs, with keys that make the running maximum jump on the way."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    q, k, v = (torch.randn(B, H, N, d, device="cuda", generator=g) for _ in range(3))
    k[:, :, N // 3:N // 3 + 9] *= 12.0
    k[:, :, N // 2:N // 2 + 5] *= 25.0
    return tuple(x.bfloat16() for x in (q, k, v))


# 2 x 12 heads: 240 query blocks in items of two, 384 in items of four, both with a ragged end
@pytest.mark.parametrize("N,d", [(64 * 9 + 17, 64), (64 * 9 + 50, 128), (64 * 15 + 5, 64), (64 * 15 + 63, 128)])
def test_options_with_several_blocks_per_item(N, d):
    """Layout, alignment, forced blocks, thresholds, scale, estimator and routing of the kernel with several query blocks per
    CTA, against the other implementation and against itself."""
    from paper_2607_24027_b200 import binding as sb
    B, H = 2, 12
    q, k, v = _many_blocks(B, H, N, d, N)
    nq = -(-N // 64)
    forced = np.zeros(nq, dtype=np.uint8)
    forced[[1, nq - 1]] = 1
    tau = torch.randn(B, H, nq, device="cuda") * 0.05
    tau[0, 0, 0], tau[1, 3, nq - 1] = float("inf"), -float("inf")
    for kw in [dict(), dict(forced=forced), dict(tau_override=tau), dict(scale=0.3), dict(estimator=sb.SOL_EST_DIAGONAL),
               dict(mode=sb.SOL_MODE_EXACT_ONLY, forced=forced)]:
        out, counts, mask, _ = hp.run_gpu(q, k, v, 64, 0.4, **kw)
        ref, counts2, mask2, _ = hp.run_gpu(q, k, v, 64, 0.4, impl=sb.SOL_IMPL_MMA_SYNC, **kw)
        assert np.array_equal(counts.cpu().numpy(), mask.sum(axis=-1))
        same = (mask == mask2).all(axis=-1)                        # a score within rounding of its threshold may differ
        assert same.mean() > 0.995, kw
        rows = torch.from_numpy(np.repeat(same, 64, axis=-1)[..., :N]).cuda()
        # bf16 weights and outputs on both sides: two tolerances of one side, in spacings of the value above 2
        err, bound = (out.float() - ref.float()).abs()[rows], torch.clamp(ref.float().abs()[rows] * 2e-2, min=2 * hp.MAX_ABS)
        assert bool((err <= bound).all()), (kw, float(err.max()))
        if "forced" in kw:
            assert mask[..., forced.astype(bool)].all()
    base, counts, mask, ws = hp.run_gpu(q, k, v, 64, 0.4)
    t = [x.transpose(1, 2).contiguous() for x in (q, k, v)]
    out, counts2, _, _ = hp.run_gpu(*t, 64, 0.4, layout=sb.SOL_LAYOUT_BNHD)
    assert torch.equal(out.transpose(1, 2), base) and torch.equal(counts2, counts)
    store = torch.empty(base.numel() + 8, dtype=base.dtype, device="cuda")
    out = store[8:].view(base.shape)                               # 16-byte aligned, not 32
    sb.sol_attn_forward_ex(q, k, v, out, ws, 64, 64, threshold=0.4)
    assert torch.equal(out, base)
    out, _, mask2, _ = hp.run_gpu(q, k, v, 64, 0.4, routing=sb.SOL_ROUTING_PREPASS)
    same = (mask == mask2).all(axis=-1)
    assert same.mean() > 0.995
    rows = torch.from_numpy(np.repeat(same, 64, axis=-1)[..., :N]).cuda()
    assert torch.equal(out[rows], base[rows])                      # the same tiles in the same order


def test_not_finite_inputs_with_several_blocks_per_item():
    """A key that scores -inf takes no part; a NaN query is a zero row, and its neighbours in the tile do not notice."""
    from paper_2607_24027_b200 import binding as sb
    B, H, N, d = 1, 24, 64 * 16 - 10, 64
    q, k, v = _many_blocks(B, H, N, d, 9)
    q[..., 0] = 1.0
    k[:, :, 200, :] = 0.0
    k[:, :, 200, 0] = -float("inf")
    q[:, 3, 77] = float("nan")
    out, counts, _, _ = hp.run_gpu(q, k, v, 64, 0.0, mode=sb.SOL_MODE_EXACT_ONLY, forced=np.ones(16))   # every block exact
    assert bool((counts == 16).all())
    keep = torch.ones(N, dtype=torch.bool, device="cuda")
    keep[200] = False
    ref = torch.nn.functional.scaled_dot_product_attention(q.double(), k[:, :, keep].double(), v[:, :, keep].double())
    good = torch.ones(H, N, dtype=torch.bool, device="cuda")
    good[3, 77] = False
    err = (out[0].double() - ref[0]).abs()[good]
    assert bool((err <= torch.clamp(ref[0][good].abs() * 1e-2, min=hp.MAX_ABS)).all()), float(err.max())
    assert bool((out[0][~good] == 0).all())


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("routing", ["fused", "prepass"])
def test_bounded_wait_runs_out(d, routing):
    """A value tile's slot that is never handed back, in a ring of four, with 24 tiles per work item: the waits run out after
    about a millisecond, every role drains what it has in flight, and the same workspace serves the next call."""
    from paper_2607_24027_b200 import binding as sb
    H, N = 40, 64 * 24
    q, k, v = _many_blocks(1, H, N, d, 11)
    route = sb.SOL_ROUTING_PREPASS if routing == "prepass" else sb.SOL_ROUTING_FUSED
    good, counts, _, ws = hp.run_gpu(q, k, v, 64, -float("inf"), routing=route)
    assert bool((counts == 24).all())
    out, mask = torch.empty_like(q), torch.zeros(1, H, 24, 1, dtype=torch.int32, device="cuda")
    sb.sol_attn_debug_set_wait(2_000_000, 1)
    try:
        sb.sol_attn_forward_ex(q, k, v, out, ws, 64, 64, threshold=-float("inf"), mask_out=mask, routing=route)
        torch.cuda.synchronize()
        detail = int(ws.buf[:8].view(torch.int32)[1].item())
        sb.sol_attn_bind_workspace(ws)
        st = sb.sol_attn_read_device_status()
    finally:
        sb.sol_attn_debug_set_wait(0, -1)
    assert st == sb.SOL_ERR_DEVICE_TIMEOUT, sb.status_string(st)
    assert detail != 0                                       # where the first wait gave up
    again, counts, _, _ = hp.run_gpu(q, k, v, 64, -float("inf"), routing=route, ws=ws)
    assert torch.equal(again, good) and bool((counts == 24).all())
