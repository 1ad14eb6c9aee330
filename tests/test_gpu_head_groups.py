"""Heads are independent: what a head gets does not depend on the heads it is called with."""
import pytest
import torch

from tests import helpers as hp

pytestmark = pytest.mark.gpu


def _qkv(H, N, d, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return tuple(torch.randn(1, H, N, d, device="cuda", generator=g).bfloat16() for _ in range(3))


@pytest.mark.parametrize("d,n_blocks", [(64, 130), (128, 130), (128, 311), (128, 32)])
def test_thresholds_of_a_head(d, n_blocks):
    """Sums split over one to eight CTAs per head, by the number of heads: the same bits."""
    from paper_2607_24027_b200 import binding as sb
    block, N = 16, 16 * n_blocks - 7
    q, k, v = _qkv(160, N, d, n_blocks)

    def thresholds(first, n):
        ws = sb.make_workspace(1, n, N, d, block, block)
        sb.sol_attn_bind_workspace(ws)
        sb.sol_attn_pool(*(x[:, first:first + n] for x in (q, k, v)), block, block, 0.6)
        return torch.stack([ws.mu, ws.sigma, ws.tau])

    whole = thresholds(0, 160)
    for first, n in [(0, 100), (50, 80), (3, 48), (100, 40), (7, 30), (9, 25), (11, 20), (140, 14), (159, 1)]:
        assert torch.equal(thresholds(first, n), whole[:, :, first:first + n]), (first, n)


@pytest.mark.parametrize("H,N,d,block,per", [(10, 64 * 140, 64, 64, 3), (6, 128 * 131, 128, 128, 1), (6, 64 * 30 - 9, 128, 64, 2)])
def test_host_path_groups(monkeypatch, H, N, d, block, per):
    """More key blocks than the one-pass threshold kernel takes, and groups of so few blocks that a call of their own would
    go to another kernel: the host path in groups of heads returns what one call returns, bit for bit."""
    from paper_2607_24027_b200 import binding as sb
    q, k, v = _qkv(H, N, d, N)
    ref, counts_ref, _, _ = hp.run_gpu(q, k, v, block, 0.8)
    ws = sb.make_workspace(1, H, N, d, block, block)
    sb.sol_attn_bind_workspace(ws)
    host = [x.cpu().pin_memory() for x in (q, k, v)] + [torch.zeros(q.shape, dtype=q.dtype).pin_memory()]
    device = [torch.empty_like(q) for _ in range(4)]
    monkeypatch.setenv("SOL_ATTN_HOST_GROUP_BYTES", str(N * d * 2 * per))
    sb.sol_attn_forward_host(*host, *device, block, block, 0.8)
    torch.cuda.synchronize()
    assert torch.equal(host[3].view(torch.int16), ref.cpu().view(torch.int16))
    assert torch.equal(ws.counts, counts_ref)
