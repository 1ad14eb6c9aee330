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
