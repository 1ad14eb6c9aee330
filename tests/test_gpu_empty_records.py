"""Keep-or-drop calls in which many chunks of key blocks hold nothing for a query block."""
import pytest
import torch

from tests import helpers as hp

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H,N,d,block", [(40, 128 * 24, 64, 128), (40, 64 * 100, 64, 64), (1, 128 * 900, 64, 128)])
@pytest.mark.parametrize("prepass", [False, True])
def test_nothing_routed(H, N, d, block, prepass):
    """More records without a tile in a row than the ring of a CTA holds, over work items and within one."""
    from paper_2607_24027_b200 import binding as sb
    g = torch.Generator(device="cuda")
    g.manual_seed(1)
    q, k, v = (torch.randn(1, H, N, d, device="cuda", generator=g).bfloat16() for _ in range(3))
    out, counts, _, _ = hp.run_gpu(q, k, v, block, float("inf"), mode=sb.SOL_MODE_EXACT_ONLY,
                                   routing=sb.SOL_ROUTING_PREPASS if prepass else sb.SOL_ROUTING_FUSED)
    assert bool((out == 0).all()) and int(counts.sum()) == 0


@pytest.mark.parametrize("block,N", [(128, 128 * 900), (64, 64 * 500)])
def test_few_blocks_far_apart(block, N):
    """One or two key blocks routed among seven chunks: the same result as the other implementation."""
    from paper_2607_24027_b200 import binding as sb
    g = torch.Generator(device="cuda")
    g.manual_seed(2)
    q, k, v = (torch.randn(1, 1, N, 64, device="cuda", generator=g).bfloat16() for _ in range(3))
    out, counts, mask, _ = hp.run_gpu(q, k, v, block, 3.2, mode=sb.SOL_MODE_EXACT_ONLY)
    ref, counts2, mask2, _ = hp.run_gpu(q, k, v, block, 3.2, mode=sb.SOL_MODE_EXACT_ONLY, impl=sb.SOL_IMPL_MMA_SYNC)
    assert 0 < int(counts.sum()) < 4 * counts.numel()
    same = torch.from_numpy((mask == mask2).all(axis=-1)[0, 0]).cuda().repeat_interleave(block)[:N]
    assert float(same.float().mean()) > 0.99
    some = (counts[0, 0] > 0).repeat_interleave(block)[:N] & same
    assert float((out[0, 0].float() - ref[0, 0].float())[some].abs().max()) <= 2 * hp.MAX_ABS
