"""Routing bits next to the cutoff: scores of one product, where every product of bf16 parts decides bits, scores of many
products of one sign, and numbers whose parts or products leave the range of fp32."""
import math

import numpy as np
import pytest
import torch

# What the products of parts may differ by, relative to a score that is one product: the three that are left out 2^-24, the two
# additions at the end 2^-24 each, those of the small terms (towards zero, at sums below 2^-7 of the score) less than 2^-28.
ONE_PRODUCT = 4 * 2.0 ** -24
SIX = [(0, 1), (1, 0), (1, 1), (0, 2), (2, 0), (0, 0)]


def _away(s, distance, up):
    """fp32 cutoffs at least ``distance`` from s, above it or below."""
    t = (s + np.where(up, distance, -distance)).astype(np.float32)
    near = np.abs(t.astype(np.float64) - s) < distance
    return np.where(near, np.nextafter(t, np.where(up, np.float32(np.inf), np.float32(-np.inf))), t).astype(np.float32)


def _one_product(heads, nq, nk, d, seed, q_size=1.0, k_size=1.0):
    """Queries with one channel that is not zero, keys of 24-bit numbers, and per query a cutoff next to its score with one key."""
    rng = np.random.default_rng(seed)
    number = lambda *shape: (rng.uniform(1, 2, shape) * rng.choice([-1, 1], shape)).astype(np.float32)
    per_channel = 2.0 ** rng.integers(-6, 7, d)                   # magnitudes that differ from channel to channel
    q, k = np.zeros((heads, nq, d), np.float32), (number(heads, nk, d) * (k_size * per_channel)).astype(np.float32)
    i = np.arange(nq)
    q[:, i, i * 37 % d] = (number(heads, nq) * (q_size / per_channel[i * 37 % d])).astype(np.float32)
    s = q.astype(np.float64) @ k.astype(np.float64).transpose(0, 2, 1)
    at = s[:, i, i * 7 % nk]
    tau = _away(at, ONE_PRODUCT * np.abs(at), (i // 3) % 2 == 0)
    near = np.abs(s - tau[:, :, None]) < ONE_PRODUCT * np.abs(s)
    assert not near[:, i, i * 7 % nk].any()
    return q, k, tau, s, near


def _parts(x):
    out = []
    for _ in range(3):
        bits = x.view(np.uint32).astype(np.uint64)
        part = ((bits + 0x7fff + (bits >> 16 & 1)) >> 16 << 16).astype(np.uint32).view(np.float32)
        out.append(part.astype(np.float64))
        x = (x - part).astype(np.float32)
    return out


@pytest.mark.parametrize("left_out", [None, *range(5)])
def test_every_product_decides_bits(left_out):
    """The cutoffs of ``_one_product`` show each of the five small products where it is missing."""
    q, k, tau, s, near = _one_product(2, 129, 129, 64, 1)
    i = np.arange(129)
    x, y = (_parts(v) for v in (q[:, i, i * 37 % 64][:, :, None], k[:, :, i * 37 % 64].transpose(0, 2, 1)))
    kept = [p for n, p in enumerate(SIX) if n != left_out]
    small = sum(x[a] * y[b] for a, b in kept if a + b)
    score = (x[0] * y[0]).astype(np.float32) + small.astype(np.float32)
    wrong = ((score > tau[:, :, None]) != (s > tau[:, :, None])) & ~near
    assert wrong.any() == (left_out is not None)


def _bits(q, k, tau):
    from paper_2607_24027_b200 import binding as sb
    heads, nq, d = q.shape
    assert nq == k.shape[1]                        # one block size for both
    N = nq * 64
    ws = sb.make_workspace(1, heads, N, d, 64, 64)
    sb.sol_attn_bind_workspace(ws)
    ws.buf[:64].fill_(90)                          # the status words, which are not this call's
    ws.qbar.copy_(torch.from_numpy(q)), ws.kc.copy_(torch.from_numpy(k))
    mask = torch.full((1, heads, nq, sb.mask_words(nq)), -1, dtype=torch.int32, device="cuda")
    tau = torch.from_numpy(np.ascontiguousarray(tau))[None].cuda()
    sb.sol_attn_route_mask(1, heads, N, d, 64, 64, mask, scale=1.0, tau_override=tau)
    assert bool((ws.buf[:64] == 90).all())
    bits = (mask[0].long()[..., None] >> torch.arange(32, device="cuda")) & 1
    return bits.flatten(-2).bool()[..., :nq].cpu().numpy()


@pytest.mark.gpu
@pytest.mark.parametrize("n,d", [(31, 64), (129, 64), (129, 128), (257, 128)])
# (as they are met; a query and a key so small that products of their parts, or parts, are below what fp32 and bf16 hold)
@pytest.mark.parametrize("q_size,k_size", [(1.0, 1.0), (2.0 ** -70, 2.0 ** -40), (2.0 ** -118, 2.0 ** 20)])
def test_one_product(n, d, q_size, k_size):
    q, k, tau, s, near = _one_product(2, n, n, d, n + d, q_size, k_size)
    assert bool(((_bits(q, k, tau) == (s > tau[:, :, None])) | near).all())


@pytest.mark.gpu
@pytest.mark.parametrize("n,d", [(129, 64), (257, 128)])
def test_products_of_one_sign(n, d):
    """All products positive: what the tensor core rounds off when it adds goes one way.  2 sqrt(d) 2^-24 of the sum, as for
    products of both signs; the d / 16 additions to an accumulator lose 2^-23 of it each at the most."""
    rng = np.random.default_rng(n)
    q, k = ((3 + 0.1 * rng.standard_normal((2, n, d))).astype(np.float32) for _ in range(2))
    s = q.astype(np.float64) @ k.astype(np.float64).transpose(0, 2, 1)
    i = np.arange(n)
    margin = 2 * math.sqrt(d) * 2.0 ** -24
    at = s[:, i, i * 7 % n]
    tau = _away(at, margin * at, (i // 3) % 2 == 0)
    near = np.abs(s - tau[:, :, None]) < margin * s
    assert bool(((_bits(q, k, tau) == (s > tau[:, :, None])) | near).all())


def _fma_scores(q, k):
    """Even and odd channels summed in fp32, one FMA after the other, and then added (fp64 holds each product and sum here to
    far below an fp32 rounding)."""
    chains = []
    with np.errstate(all="ignore"):
        for first in (0, 1):
            acc = np.zeros((q.shape[0], q.shape[1], k.shape[1]), np.float32)
            for c in range(first, q.shape[2], 2):
                acc = (q[:, :, None, c].astype(np.float64) * k[:, None, :, c] + acc).astype(np.float32)
            chains.append(acc)
        return chains[0] + chains[1]


@pytest.mark.gpu
@pytest.mark.parametrize("n,d", [(65, 64), (129, 128)])
def test_scores_beyond_fp32(n, d):
    """Finite numbers whose products overflow compare as sums of FMAs do: infinities of either sign, and NaN where two meet."""
    rng = np.random.default_rng(d)
    q, k = (rng.standard_normal((3, n, d)).astype(np.float32) for _ in range(2))
    k = np.abs(k)                                   # (the one channel below decides)
    big = np.float32(1.0039 * 2.0 ** 64)            # its first and second parts have opposite signs
    q[0, ::2, 5], k[0, 1::3, 5] = big, big
    q[1, ::2, 5], k[1, 1::3, 5] = -big, big
    q[2, ::3, 4], q[2, ::3, 7], k[2, 1::3, 4], k[2, 1::3, 7] = big, -big, big, big   # + inf and - inf in the two chains
    q[2, 1::3, 9] = np.finfo(np.float32).max        # rounds up to an infinite part
    tau = (0.1 * rng.standard_normal((3, n))).astype(np.float32)
    s = _fma_scores(q, k)
    assert np.isposinf(s).any() and np.isneginf(s).any() and np.isnan(s).any()
    size = np.abs(q).astype(np.float64) @ np.abs(k).astype(np.float64).transpose(0, 2, 1)
    near = (np.abs(s.astype(np.float64) - tau[:, :, None]) <= 2 * math.sqrt(d) * 2.0 ** -24 * size) & np.isfinite(s)
    assert not near[~np.isfinite(s)].any() and near.mean() < 0.5
    assert bool(((_bits(q, k, tau) == (s > tau[:, :, None])) | near).all())


@pytest.mark.gpu
@pytest.mark.parametrize("n,d,withhold", [(129, 64, 0), (129, 128, 0), (129, 128, 1)])
def test_without_a_completion_signal(n, d, withhold):
    """The wait for the tensor core runs out after about a millisecond: the bits come from FMAs, the tensor memory goes back
    behind the MMAs, and the next call is a normal one."""
    from paper_2607_24027_b200 import binding as sb
    q, k, tau, s, near = _one_product(2, n, n, d, n + d)
    want = s > tau[:, :, None]
    sb.sol_attn_debug_set_wait(2_000_000, withhold)
    try:
        bits = _bits(q, k, tau)
        torch.cuda.synchronize()
    finally:
        sb.sol_attn_debug_set_wait(0, -1)
    assert bool(((bits == want) | near).all())
    assert bool(((_bits(q, k, tau) == want) | near).all())
