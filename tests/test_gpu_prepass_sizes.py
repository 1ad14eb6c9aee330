"""Thresholds, routing bits and materialised routing at the sizes where their kernels change hands or tiles end."""
import math

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sb():
    from paper_2607_24027_b200 import binding
    binding.lib()
    return binding


def _pooled(BH, N, d, block, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    q, k, v = (torch.randn(1, BH, N, d, device="cuda", generator=g).bfloat16() for _ in range(3))
    return q, k, v


# Nk: one block, sizes at which the one-pass kernel's shared memory is just below and above 48 KB, the sizes next to its 128, row
# steps of 32 / 64 / 88 per CTA of a cluster, ragged chunks of keys, and clusters of 8 (up to 14 heads), 6 (20), 5 (25, 48), 4 (30),
# 3 (40, 80), 2 (60, 100) and 1 (400 heads)
@pytest.mark.parametrize("BH,n_blocks,d", [(1, 1, 64), (3, 17, 128), (2, 66, 128), (2, 73, 128), (2, 90, 128), (2, 92, 128), (2, 128, 64), (2, 128, 128), (2, 129, 64), (2, 129, 128),
                                           (3, 300, 128), (40, 260, 128), (40, 591, 64), (400, 130, 64), (1, 1500, 128),
                                           (14, 161, 64), (20, 193, 128), (25, 160, 128), (30, 131, 64), (48, 140, 128), (60, 150, 64),
                                           (80, 133, 128), (100, 191, 64), (400, 129, 128)])
@pytest.mark.parametrize("estimator", ["moments", "diagonal"])
def test_thresholds(sb, BH, n_blocks, d, estimator):
    block = 64 if n_blocks < 1000 else 16
    N = n_blocks * block - 5
    q, k, v = _pooled(BH, N, d, block, n_blocks)
    ws = sb.make_workspace(1, BH, N, d, block, block)
    sb.sol_attn_bind_workspace(ws)
    sb.sol_attn_pool(q, k, v, block, block, 0.7)
    sb.sol_attn_thresholds(1, BH, N, d, block, block, 0.7,
                           estimator=sb.SOL_EST_DIAGONAL if estimator == "diagonal" else sb.SOL_EST_MOMENTS)
    qb, kc = ws.qbar[0].double() / math.sqrt(d), ws.kc[0].double()
    s = qb @ kc.transpose(1, 2)
    mu = s.mean(dim=2)
    if estimator == "diagonal":
        sigma = (qb.square() @ kc.var(dim=1, correction=0)[:, :, None])[:, :, 0].sqrt()
    else:
        sigma = s.var(dim=2, correction=0).sqrt()
    # fp32 sums of up to 1500 terms and of d products: a few 1e-6 of the largest score at the very most
    tol = 4e-6 * float(s.abs().max()) + 1e-9
    assert float((ws.mu[0] - mu).abs().max()) <= tol
    assert float((ws.sigma[0] - sigma).abs().max()) <= tol
    assert float((ws.tau[0] - (mu + 0.7 * sigma)).abs().max()) <= 2 * tol


@pytest.mark.parametrize("BH,nq,nk,d", [(1, 1, 1, 32), (2, 127, 63, 64), (2, 129, 65, 128), (3, 128, 64, 96), (1, 200, 1024, 64),
                                        (1, 5, 1025, 64), (2, 33, 32, 128), (2, 33, 33, 128), (1, 9, 513, 64)])
@pytest.mark.parametrize("aligned", [True, False])
def test_materialised_order(sb, BH, nq, nk, d, aligned):
    g = torch.Generator(device="cuda")
    g.manual_seed(nk)
    # whole numbers with many ties (and zeros of both signs): products and sums are exact, so the order is too
    def whole(n):
        flat = torch.randint(-2, 3, (BH * n * d + 1,), device="cuda", generator=g).float()
        x = flat[:-1] if aligned else flat[1:]
        return x.view(1, BH, n, d)
    qb, kc = whole(nq), whole(nk)
    pm = torch.empty(1, BH, nq, nk, device="cuda")
    order = torch.empty(1, BH, nq, nk, dtype=torch.int32, device="cuda")
    counts = torch.empty(1, BH, nq, dtype=torch.int32, device="cuda")
    tau = torch.empty(1, BH, nq, device="cuda")
    ref = (qb[0].double() @ kc[0].double().transpose(1, 2)).cpu().numpy()
    want = np.argsort(-ref, axis=-1, kind="stable")                # higher score first, lower index on ties
    for c in {0, 1, nk // 2, nk - 1, nk}:
        sb.sol_attn_route_materialized(qb, kc, sb.SOL_ROUTE_TOPK, c, pm, tau, order=order, counts=counts, scale=1.0)
        assert np.array_equal(pm[0].cpu().numpy().astype(np.float64), ref)
        assert np.array_equal(order[0].cpu().numpy(), want)
        assert bool((counts == c).all())
        top = np.take_along_axis(ref, want, axis=-1)
        t = np.full(ref.shape[:2], np.inf if c == 0 else -np.inf) if c in (0, nk) else (top[..., c - 1] + top[..., c]) / 2
        assert np.array_equal(tau[0].cpu().numpy().astype(np.float64), t)


@pytest.mark.parametrize("nk", [33, 250, 256, 700, 1024, 1500, 5000])
def test_top_p_of_one_ends_with_the_mass(sb, nk):
    """p = 1 keeps the blocks that have any share: the running sum of a lane may round differently from the scan over the
    lanes, which must not make the row miss its end and keep everything."""
    rows, d = 400, 32
    rng = np.random.default_rng(nk)
    some = rng.integers(1, nk, rows)                               # blocks with mass; the others' exponentials are zero
    scores = np.where(np.arange(nk) < some[:, None], rng.uniform(-3, 3, (rows, nk)), -1e4).astype(np.float32)
    for row in scores:
        rng.shuffle(row)
    qb, kc = torch.zeros(1, rows, 1, d), torch.zeros(1, rows, nk, d)
    qb[..., 0] = 1.0
    kc[0, :, :, 0] = torch.from_numpy(scores)                     # one row of scores per head
    pm, counts, tau = torch.empty(1, rows, 1, nk), torch.empty(1, rows, 1, dtype=torch.int32), torch.empty(1, rows, 1)
    qb, kc, pm, counts, tau = (x.cuda() for x in (qb, kc, pm, counts, tau))
    sb.sol_attn_route_materialized(qb, kc, sb.SOL_ROUTE_TOPP, 1.0, pm, tau, counts=counts, scale=1.0)
    assert np.array_equal(counts.cpu().numpy()[0, :, 0], some)


@pytest.mark.parametrize("n_q,n_k", [(1, 1), (127, 63), (128, 64), (129, 65), (257, 97), (64, 591)])
def test_mask_bits(sb, n_q, n_k):
    """Bits of ragged tiles, against the same comparison in 64 bits; block_q and block_k differ so that Nq and Nk do."""
    d, H = 128, 3
    N = 16 * max(n_q, n_k)
    bq, bk = -(-N // n_q), -(-N // n_k)
    if bq > 1024 or bk > 1024:
        pytest.skip("block size limit")
    q, k, v = _pooled(H, N, d, bq, n_q)
    ws = sb.make_workspace(1, H, N, d, bq, bk)
    nq, nk = ws.view.n_q_blocks, ws.view.n_k_blocks
    sb.sol_attn_bind_workspace(ws)
    sb.sol_attn_pool(q, k, v, bq, bk, 0.5)
    words = sb.mask_words(nk)
    mask = torch.full((1, H, nq, words), -1, dtype=torch.int32, device="cuda")
    forced = torch.zeros(nk, dtype=torch.uint8, device="cuda")
    forced[nk // 2] = 1
    sb.sol_attn_route_mask(1, H, N, d, bq, bk, mask, forced_blocks=forced)
    s = (ws.qbar[0].double() @ ws.kc[0].double().transpose(1, 2)) / math.sqrt(d)
    gap = (s - ws.tau[0].double()[:, :, None]).cpu().numpy()
    bits = np.unpackbits(mask[0].cpu().numpy().view(np.uint8), axis=-1, bitorder="little").astype(bool)
    assert not bits[..., nk:].any()
    want = gap > 0
    want[..., nk // 2] = True
    clear = np.abs(gap) > 1e-5
    clear[..., nk // 2] = True
    assert np.array_equal(bits[..., :nk][clear], want[clear])
