"""Calls of different sizes from several host threads at once, each with a workspace and a stream of its own."""
import threading

import pytest
import torch

pytestmark = pytest.mark.gpu


def _together(calls, rounds):
    """Runs each call `rounds` times on a thread and a stream of its own; returns what they raised."""
    errors, gate = [], threading.Barrier(len(calls))

    def work(call):
        stream = torch.cuda.Stream()
        gate.wait()
        try:
            for _ in range(rounds):
                call(stream)
        except Exception as e:                     # noqa: BLE001
            errors.append(e)

    torch.cuda.synchronize()
    threads = [threading.Thread(target=work, args=(c,)) for c in calls]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    return errors


def test_thresholds_of_few_and_many_keys():
    """The one-pass threshold kernel needs shared memory for its keys: 128, 100, 64 and 72 of them."""
    from paper_2607_24027_b200 import binding as sb
    calls, checks = [], []
    for n_blocks in (128, 100, 64, 72):
        q, k, v = (torch.randn(1, 1, n_blocks * 64, 128, device="cuda").bfloat16() for _ in range(3))
        ws = sb.make_workspace(1, 1, n_blocks * 64, 128, 64, 64)
        out, ref = torch.empty_like(q), torch.empty_like(q)
        sb.sol_attn_forward_ex(q, k, v, ref, ws, 64, 64, threshold=0.5)
        calls.append(lambda s, a=(q, k, v, out, ws): sb.sol_attn_forward_ex(*a, 64, 64, threshold=0.5, stream=s))
        checks.append((out, ref))
    assert not _together(calls, 400)
    assert all(torch.equal(a, b) for a, b in checks)


def test_rows_of_several_lengths():
    """The sort of long proxy rows needs shared memory for the row."""
    from paper_2607_24027_b200 import binding as sb
    calls, checks = [], []
    for nk in (8192, 1500, 5000, 2048):
        qb, kc = torch.randn(1, 1, 2, 64, device="cuda"), torch.randn(1, 1, nk, 64, device="cuda")
        pm, tau, ref = torch.empty(1, 1, 2, nk, device="cuda"), torch.empty(1, 1, 2, device="cuda"), torch.empty(1, 1, 2, device="cuda")
        sb.sol_attn_route_materialized(qb, kc, sb.SOL_ROUTE_TOPK, 100, pm, ref)
        calls.append(lambda s, a=(qb, kc), m=pm, t=tau: sb.sol_attn_route_materialized(*a, sb.SOL_ROUTE_TOPK, 100, m, t, stream=s))
        checks.append((tau, ref))
    assert not _together(calls, 400)
    assert all(torch.equal(a, b) for a, b in checks)
