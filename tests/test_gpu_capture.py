"""Calls captured into a CUDA graph and replayed on new inputs: every kernel route, as the first node of a graph, behind a
memset, and behind work that another stream joins in."""
import pytest
import torch

pytestmark = pytest.mark.gpu

# H, N, d, block: one block per CTA and several per CTA of 64 tokens; thresholds in one pass and by clusters
SHAPES = {"tiny": (2, 1024, 64, 64), "b64": (24, 64 * 20, 64, 64), "b64 clusters": (4, 64 * 150 - 3, 128, 64),
          "b128": (6, 128 * 9 + 5, 128, 128), "b128 clusters": (20, 128 * 131, 64, 128)}


def _calls(sb, q, k, v, out, ws, block, mask):
    H, N, d = q.shape[1:]
    ex = lambda **kw: sb.sol_attn_forward_ex(q, k, v, out, ws, block, block, threshold=0.6, **kw)  # noqa: E731

    def calibrate():
        sb.sol_attn_bind_workspace(ws)
        sb.sol_attn_pool(q, k, v, block, block, 0.1)
        sb.sol_attn_thresholds(1, H, N, d, block, block, 0.6)
        sb.sol_attn_route_mask(1, H, N, d, block, block, mask)
        ex(skip_pool=True)

    def topk():
        sb.sol_attn_bind_workspace(ws)
        sb.sol_attn_pool(q, k, v, block, block, 0.1)
        nk = ws.view.n_k_blocks
        pm = topk.pm = torch.empty(1, H, nk, nk, device="cuda") if topk.pm is None else topk.pm
        tau = topk.tau = torch.empty(1, H, nk, device="cuda") if topk.tau is None else topk.tau
        sb.sol_attn_route_materialized(ws.qbar, ws.kc, sb.SOL_ROUTE_TOPK, 5, pm, tau)
        ex(skip_pool=True, tau_override=tau)
    topk.pm = topk.tau = None
    return {"sol": ex, "exact_only": lambda: ex(mode=sb.SOL_MODE_EXACT_ONLY), "dense": lambda: ex(mode=sb.SOL_MODE_DENSE),
            "prepass": lambda: ex(routing=sb.SOL_ROUTING_PREPASS, mask_out=mask),
            "diagonal": lambda: ex(estimator=sb.SOL_EST_DIAGONAL), "calibrate": calibrate, "topk": topk}


@pytest.mark.parametrize("shape", list(SHAPES))
@pytest.mark.parametrize("call", ["sol", "exact_only", "dense", "prepass", "diagonal", "calibrate", "topk"])
def test_replay(shape, call):
    from paper_2607_24027_b200 import binding as sb
    H, N, d, block = SHAPES[shape]
    g = torch.Generator(device="cuda")
    g.manual_seed(N)
    sets = [[torch.randn(1, H, N, d, device="cuda", generator=g).bfloat16() for _ in range(3)] for _ in range(3)]
    q, k, v = (x.clone() for x in sets[0])
    out = torch.empty_like(q)
    ws = sb.make_workspace(1, H, N, d, block, block)
    nk = ws.view.n_k_blocks
    mask = torch.zeros(1, H, nk, sb.mask_words(nk), dtype=torch.int32, device="cuda")
    run = _calls(sb, q, k, v, out, ws, block, mask)[call]
    want = []
    for s in sets:
        for x, y in zip((q, k, v), s):
            x.copy_(y)
        run()
        torch.cuda.synchronize()
        want.append((out.clone(), ws.counts.clone(), mask.clone()))
    graph, other = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    src = [x.clone() for x in sets[0]]
    with torch.cuda.graph(graph):
        # k and v arrive on another stream, q on this one: the call's first kernel has two predecessors
        other.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(other):
            k.copy_(src[1])
            v.copy_(src[2])
        q.copy_(src[0])
        torch.cuda.current_stream().wait_stream(other)
        run()
    for i in (1, 2, 0):
        for x, y in zip(src, sets[i]):
            x.copy_(y)
        out.fill_(float("nan"))
        graph.replay()
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(out, want[i][0]) and torch.equal(ws.counts, want[i][1])
        if call in ("prepass", "calibrate"):
            assert torch.equal(mask, want[i][2])
    sb.sol_attn_bind_workspace(ws)
    assert sb.sol_attn_read_device_status() == sb.SOL_OK


@pytest.mark.parametrize("shape", ["tiny", "b128 clusters"])
def test_first_kernel_behind_another_stream(shape):
    """Re-thresholding and bits as the first work behind an event: nothing of it may start before what it waits for."""
    from paper_2607_24027_b200 import binding as sb
    H, N, d, block = SHAPES[shape]
    q, k, v = (torch.randn(1, H, N, d, device="cuda").bfloat16() for _ in range(3))
    ws = sb.make_workspace(1, H, N, d, block, block)
    sb.sol_attn_bind_workspace(ws)
    sb.sol_attn_pool(q, k, v, block, block, 0.3)
    nk = ws.view.n_k_blocks
    mask, ref = (torch.zeros(1, H, nk, sb.mask_words(nk), dtype=torch.int32, device="cuda") for _ in range(2))
    sb.sol_attn_thresholds(1, H, N, d, block, block, 0.3)
    sb.sol_attn_route_mask(1, H, N, d, block, block, ref)
    kc, junk, busy = ws.kc.clone(), torch.randn_like(ws.kc), torch.randn(4096, 4096, device="cuda")
    other, stream = torch.cuda.Stream(), torch.cuda.Stream()
    for _ in range(20):
        ws.kc.copy_(junk)
        mask.zero_()
        torch.cuda.synchronize()
        with torch.cuda.stream(other):
            for _ in range(3):
                busy @ busy
            ws.kc.copy_(kc)
        stream.wait_stream(other)
        sb.sol_attn_thresholds(1, H, N, d, block, block, 0.3, stream=stream)
        sb.sol_attn_route_mask(1, H, N, d, block, block, mask, stream=stream)
        torch.cuda.synchronize()
        assert torch.equal(mask, ref)
