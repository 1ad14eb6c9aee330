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


@pytest.fixture
def short_waits():
    """A stall shows after 30 ms of cycles instead of two seconds; the longest wait of these calls is well below 1 ms."""
    from paper_2607_24027_b200 import binding as sb
    sb.sol_attn_debug_set_wait(60_000_000, -1)
    yield
    sb.sol_attn_debug_set_wait(0, -1)


@pytest.mark.parametrize("chunks,block,d", [(5, 128, 64), (8, 128, 128), (5, 64, 64)])
@pytest.mark.parametrize("prepass", [False, True])
def test_busy_chunk_before_empty_ones(chunks, block, d, prepass, short_waits):
    """Ten forced blocks at the start and nothing else: a record with tiles, then four or more without, which the router
    writes while the tiles are worked on.  The same as attention over the first ten blocks."""
    from paper_2607_24027_b200 import binding as sb
    H, nk = 2, block * chunks - 3
    N = nk * block - 5
    g = torch.Generator(device="cuda")
    g.manual_seed(3)
    q, k, v = (torch.randn(1, H, N, d, device="cuda", generator=g).bfloat16() for _ in range(3))
    forced = torch.zeros(nk, dtype=torch.uint8)
    forced[:10] = 1
    out, counts, mask, _ = hp.run_gpu(q, k, v, block, float("inf"), mode=sb.SOL_MODE_EXACT_ONLY, forced=forced.numpy(),
                                      routing=sb.SOL_ROUTING_PREPASS if prepass else sb.SOL_ROUTING_FUSED)
    assert bool((counts == 10).all())
    some = torch.randperm(N, generator=torch.Generator().manual_seed(4))[:4096].cuda()
    keys = slice(0, 10 * block)
    ref = torch.nn.functional.scaled_dot_product_attention(q[:, :, some].double(), k[:, :, keys].double(), v[:, :, keys].double())
    assert float((out[:, :, some].double() - ref).abs().max()) <= hp.MAX_ABS
    assert bool(torch.isfinite(out).all())


@pytest.mark.parametrize("block,d", [(128, 128), (64, 64)])
@pytest.mark.parametrize("prepass", [False, True])
def test_busy_items_between_empty_ones(block, d, prepass, short_waits):
    """One query block in seven routes ten blocks or all of them, the others nothing: the same as the other implementation."""
    from paper_2607_24027_b200 import binding as sb
    H, nk = 16, 60
    N = nk * block - 40
    g = torch.Generator(device="cuda")
    g.manual_seed(5)
    q, k, v = (torch.randn(1, H, N, d, device="cuda", generator=g).bfloat16() for _ in range(3))
    ws = sb.make_workspace(1, H, N, d, block, block)
    sb.sol_attn_bind_workspace(ws)
    sb.sol_attn_pool(q, k, v, block, block, 0.0)
    top = torch.empty(1, H, nk, device="cuda")
    sb.sol_attn_route_materialized(ws.qbar, ws.kc, sb.SOL_ROUTE_TOPK, 10, torch.empty(1, H, nk, nk, device="cuda"), top)
    tau = torch.full_like(top, float("inf"))
    tau[..., ::7] = top[..., ::7]
    tau[..., 3::21] = -float("inf")
    out, counts, _, _ = hp.run_gpu(q, k, v, block, 0.0, mode=sb.SOL_MODE_EXACT_ONLY, tau_override=tau, skip_pool=True, ws=ws,
                                   routing=sb.SOL_ROUTING_PREPASS if prepass else sb.SOL_ROUTING_FUSED)
    ref, counts2, _, _ = hp.run_gpu(q, k, v, block, 0.0, mode=sb.SOL_MODE_EXACT_ONLY, tau_override=tau, skip_pool=True, ws=ws,
                                    impl=sb.SOL_IMPL_MMA_SYNC)
    assert bool((counts[..., 3::21] == nk).all()) and int((counts > 0).sum()) < counts.numel() // 4
    same = (counts == counts2)[0].repeat_interleave(block, dim=1)[:, :N]      # (a tie with the cutoff may fall either way)
    assert float(same.float().mean()) > 0.99
    assert bool((out[0][(counts[0] == 0).repeat_interleave(block, dim=1)[:, :N]] == 0).all())
    some = same & (counts[0] > 0).repeat_interleave(block, dim=1)[:, :N]
    assert float((out[0].float() - ref[0].float())[some].abs().max()) <= 2 * hp.MAX_ABS
