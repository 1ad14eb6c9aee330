"""Routing bits from products of bf16 parts: the edges of the 128 x 128 tiles, and inputs that have no parts."""
import math

import pytest
import torch

pytestmark = pytest.mark.gpu


# blocks of queries and keys below, at and above one tile, half a tile (a thread's share of the columns) and a 32-bit word
@pytest.mark.parametrize("block_q,block_k,N,d", [(64, 64, 1, 64), (64, 64, 64 * 31, 128), (64, 64, 64 * 65 - 3, 64), (64, 64, 64 * 127, 128),
                                                 (64, 64, 64 * 129 - 63, 64), (32, 64, 32 * 257, 128), (128, 32, 128 * 33 - 1, 128)])
@pytest.mark.parametrize("special", [False, True])
def test_bits(block_q, block_k, N, d, special):
    """The score in 64 bits against the cutoff, except within a few roundings of it: fp32 sums of d products, 2 sqrt(d) 2^-24 of
    the sum of their magnitudes at the most.  Infinities and NaN compare as the fp32 products do."""
    from paper_2607_24027_b200 import binding as sb
    H = 3
    g = torch.Generator(device="cuda")
    g.manual_seed(N + d)
    q, k, v = (torch.randn(1, H, N, d, device="cuda", generator=g).bfloat16() for _ in range(3))
    if special:
        k[0, 0, 0, 5], k[0, 1, N // 2, 7], q[0, 1, N - 1, 0] = math.inf, math.nan, -math.inf
    ws = sb.make_workspace(1, H, N, d, block_q, block_k)
    ws.buf[:64].zero_()                          # (the status words: pooling alone leaves them as they are)
    sb.sol_attn_bind_workspace(ws)
    sb.sol_attn_pool(q, k, v, block_q, block_k, 0.0)
    nq, nk = ws.view.n_q_blocks, ws.view.n_k_blocks
    tau = torch.randn(1, H, nq, device="cuda", generator=g) * 0.02
    forced = torch.zeros(nk, dtype=torch.uint8, device="cuda")
    forced[nk // 2] = 1
    words = sb.mask_words(nk)
    mask = torch.full((1, H, nq, words), -1, dtype=torch.int32, device="cuda")
    sb.sol_attn_route_mask(1, H, N, d, block_q, block_k, mask, tau_override=tau, forced_blocks=forced)
    assert sb.sol_attn_read_device_status() == sb.SOL_OK
    bits = ((mask.long()[..., None] >> torch.arange(32, device="cuda")) & 1).flatten(-2).bool()
    assert not bool(bits[..., nk:].any())
    qb, kc = ws.qbar.double(), ws.kc.double()
    products = qb[..., :, None, :] * kc[..., None, :, :]
    s, size = products.sum(-1) / math.sqrt(d), products.abs().sum(-1) / math.sqrt(d)
    want = (s > tau.double()[..., None]) | forced.bool()
    near = ((s - tau.double()[..., None]).abs() <= 2 * math.sqrt(d) * 2.0 ** -24 * size) & size.isfinite()
    assert bool(((bits[..., :nk] == want) | near).all())
    assert float(near.double().mean()) < 0.01
