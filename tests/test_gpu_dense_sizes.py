"""The dense kernel (two query tiles per CTA): item and tile edges, layouts, counts and mask, and its bounded waits."""
import numpy as np
import pytest
import torch

from tests import helpers as hp

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sb():
    from paper_2607_24027_b200 import binding
    binding.lib()
    return binding


def _qkv(B, H, N, d, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return tuple(torch.randn(B, H, N, d, device="cuda", generator=g).bfloat16() for _ in range(3))


# more than 148 tiles of 128 rows over all heads; one key tile, two, five and more than the ring holds; the last item
# with one tile, the last tile with 1, 64, 127 and 128 rows; one and several items per CTA
@pytest.mark.parametrize("B,H,N,d", [(1, 149, 128, 128), (2, 100, 1, 64), (1, 75, 129, 128), (1, 60, 320, 64), (2, 40, 511, 128),
                                     (1, 40, 640, 128), (3, 50, 769, 64), (1, 40, 1700, 128), (1, 300, 257, 128)])
@pytest.mark.parametrize("block", [64, 128])
def test_sizes(sb, B, H, N, d, block):
    q, k, v = _qkv(B, H, N, d, N + d)
    if N > 400:
        k[:, :, 300:310] *= 40.0                   # maxima that grow along the keys: the accumulator is rescaled
    out, counts, mask, _ = hp.run_gpu(q, k, v, block, 0.0, mode=sb.SOL_MODE_DENSE)
    ref = torch.nn.functional.scaled_dot_product_attention(q.double(), k.double(), v.double())
    err = (out.double() - ref).abs()
    # P and the output are rounded to bf16: 1e-2, or 1.28 spacings of the output above 2, as for every kernel here
    assert bool((err <= torch.clamp(ref.abs() * 1e-2, min=hp.MAX_ABS)).all()), float(err.max())
    assert float(err.norm() / ref.norm()) <= 5e-3
    assert bool((counts == -(-N // block)).all()) and bool(mask.all())


def test_layout_and_unaligned_rows(sb):
    B, H, N, d = 1, 40, 700, 128
    q, k, v = _qkv(B, H, N, d, 3)
    a, _, _, _ = hp.run_gpu(q, k, v, 128, 0.0, mode=sb.SOL_MODE_DENSE)
    t = [x.transpose(1, 2).contiguous() for x in (q, k, v)]
    b, _, _, _ = hp.run_gpu(*t, 128, 0.0, mode=sb.SOL_MODE_DENSE, layout=sb.SOL_LAYOUT_BNHD)
    assert torch.equal(a, b.transpose(1, 2))
    store = torch.empty(a.numel() + 8, dtype=a.dtype, device="cuda")
    out = store[8:].view(a.shape)                  # 16-byte aligned, not 32
    ws = sb.make_workspace(B, H, N, d, 128, 128)
    sb.sol_attn_forward_ex(q, k, v, out, ws, 128, 128, mode=sb.SOL_MODE_DENSE)
    assert torch.equal(out, a)


def test_infinite_and_nan_inputs(sb):
    """A key that scores -inf everywhere takes no part; a NaN query has no finite logit, so its row is zero, and the
    rows beside it in the tile do not notice."""
    B, H, N, d = 1, 40, 600, 64
    q, k, v = _qkv(B, H, N, d, 4)
    q[..., 0] = 1.0
    k[:, :, 200, :] = 0.0
    k[:, :, 200, 0] = -float("inf")                # weight 0 for every query
    q[:, 3, 77] = float("nan")
    out, _, _, _ = hp.run_gpu(q, k, v, 64, 0.0, mode=sb.SOL_MODE_DENSE)
    keep = torch.ones(N, dtype=torch.bool, device="cuda")
    keep[200] = False
    ref = torch.nn.functional.scaled_dot_product_attention(q.double(), k[:, :, keep].double(), v[:, :, keep].double())
    bad = torch.zeros(H, N, dtype=torch.bool, device="cuda")
    bad[3, 77] = True
    assert bool(torch.isfinite(out[0][~bad]).all())
    assert float((out[0][~bad].double() - ref[0][~bad]).abs().max()) <= hp.MAX_ABS
    assert bool((out[0][bad] == 0).all())


def test_bounded_wait_runs_out(sb):
    q, k, v = _qkv(1, 40, 1700, 128, 5)
    ws = sb.make_workspace(1, 40, 1700, 128, 128, 128)
    out = torch.empty_like(q)
    good, _, _, _ = hp.run_gpu(q, k, v, 128, 0.0, mode=sb.SOL_MODE_DENSE)
    sb.sol_attn_debug_set_wait(2_000_000, 1)
    try:
        sb.sol_attn_forward_ex(q, k, v, out, ws, 128, 128, mode=sb.SOL_MODE_DENSE)
        torch.cuda.synchronize()
        sb.sol_attn_bind_workspace(ws)
        st = sb.sol_attn_read_device_status()
    finally:
        sb.sol_attn_debug_set_wait(0, -1)
    assert st == sb.SOL_ERR_DEVICE_TIMEOUT, sb.status_string(st)
    again, _, _, _ = hp.run_gpu(q, k, v, 128, 0.0, mode=sb.SOL_MODE_DENSE, ws=ws)
    assert torch.equal(again, good)
