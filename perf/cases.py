"""The calls that users of this package make, as cases that can be timed.

The package computes attention for diffusion transformers: images, videos and video editing, over 10^3 to 7.6 * 10^4 tokens and
2 to 40 heads, in bf16, with 5 to 60 % of the key blocks exact.  The listed cases are the workloads of
``paper_2607_24027_b200.configs`` and the ways of calling the operator that its header describes; ``draw`` spreads over the same
ranges.  A case says what is called (``op``), the token grid (``frames`` x ``rows`` x ``cols``, twice that when ``edit``, plus
``text`` tokens), and the options.

    forward    sol_attn_forward: pooling, thresholds and the fused kernel
    dense      sol_attn_dense: the denoising steps and layers that a sampler keeps dense
    options    sol_attn_forward_ex with a layout, a routing, an estimator, a mode or forced blocks
    host       sol_attn_forward_host: tensors in pinned host memory
    calibrate  sol_attn_thresholds + sol_attn_route_mask: another density on tensors that are pooled already
    topk       sol_attn_pool, sol_attn_route_materialized and the fused kernel: a top-k policy drives the operator
"""
import math

import numpy as np
import torch

from paper_2607_24027_b200 import binding as sol
from paper_2607_24027_b200 import synth
from paper_2607_24027_b200.configs import load_betas

# The largest listed case; a drawn one is not larger.
_MOST_FLOPS = 4.0 * 40 * 32760.0 ** 2 * 128


def _case(op, heads, d, block, grid, density, beta, name=None, batch=1, text=0, edit=False, sinks=False, mode="sol",
          tokens_first=False, prepass=False, diagonal=False, forced=False):
    c = {"op": op, "batch": batch, "heads": heads, "d": d, "block": block, "frames": grid[0], "rows": grid[1],
         "cols": grid[2], "text": text, "edit": edit, "sinks": sinks, "density": density, "beta": beta, "mode": mode,
         "tokens_first": tokens_first, "prepass": prepass, "diagonal": diagonal, "forced": forced}
    if name:
        c["name"] = name
    return c


def listed():
    image, video480, video720 = (1, 64, 64), (21, 30, 52), (21, 45, 80)
    return [
        # the smallest configuration: launches and latency
        _case("forward", 2, 64, 64, (4, 16, 16), 0.28, 0.5979, "tiny"),
        # an image transformer, one layer of one step
        _case("forward", 24, 128, 128, image, 0.30, 0.0712, "image"),
        # the same with text tokens behind the image that stay exact, guidance as a batch of two, and q, k, v as a fused
        # projection leaves them; a ragged last block
        _case("options", 24, 128, 128, image, 0.43, -0.1936, "image_text", batch=2, text=77, tokens_first=True, forced=True),
        # the same image from and to host memory
        _case("host", 24, 128, 128, image, 0.30, 0.0712, "image_host"),
        # small heads and small blocks, an odd token count, unselected blocks dropped (the keep-or-drop ablation)
        _case("options", 16, 64, 64, (8, 31, 45), 0.20, 0.90, "small_blocks", sinks=True, mode="exact_only"),
        # 480p video, 81 frames: a sparse step, and a dense one as the first steps of a sampler are
        _case("forward", 40, 128, 128, video480, 0.25, 0.5347, "video480", sinks=True),
        _case("dense", 40, 128, 128, video480, 1.0, 0.0, "video480_dense", sinks=True),
        # 720p video, at the density of the headline and, routed by the pre-pass, at the lowest one
        _case("forward", 40, 128, 128, video720, 0.15, 1.0465, "video720", sinks=True),
        _case("options", 40, 128, 128, video720, 0.05, 2.0728, "video720_low", sinks=True, prepass=True),
        # video editing, source and target in one sequence, with the diagonal threshold estimator
        _case("options", 40, 128, 128, video480, 0.223, 1.2184, "edit", edit=True, sinks=True, diagonal=True),
        # a density search on pooled 720p tensors
        _case("calibrate", 40, 128, 128, video720, 0.15, 1.0465, "video720_calibrate", sinks=True),
        # top-k block selection at 480p
        _case("topk", 40, 128, 128, video480, 0.15, 0.0, "video480_topk", sinks=True),
    ]


def _beta(kind, density):
    """The calibrated cutoff for a density, interpolated in the workload's table."""
    table = sorted(load_betas()[kind].items())
    return round(float(np.interp(density, [r for r, _ in table], [b for _, b in table])), 4)


def _tokens(c):
    return c["frames"] * c["rows"] * c["cols"] * (2 if c["edit"] else 1) + c["text"]


def draw(rng):
    while True:
        op = rng.choice(["forward", "forward", "forward", "options", "options", "options", "dense", "host", "calibrate", "topk"])
        # the tokens over their logarithm, from a few blocks to 720p video, in a grid of roughly that many
        tokens = math.exp(rng.uniform(math.log(700), math.log(75600)))
        video = tokens > 9000 or (tokens > 2500 and rng.random() < 0.4)
        frames = rng.randint(4, 24) if video else rng.choice([1, 1, 1, 4])
        rows = max(4, round(math.sqrt(tokens / frames) * rng.uniform(0.6, 1.1)))
        cols = max(4, round(tokens / frames / rows))
        edit = video and rng.random() < 0.2
        if edit:
            frames = max(2, frames // 2)
        text = 0 if video or rng.random() < 0.5 else rng.randint(16, 512)
        d, block = rng.choice([(128, 128)] * 5 + [(64, 64), (64, 128), (128, 64)])
        heads, batch = rng.choice([2, 5, 12, 16, 24, 24, 30, 40, 40, 40]), rng.choice([1, 1, 1, 2])
        low, high, kind = (0.05, 0.5, "edit" if edit else "video720") if video else (0.2, 0.6, "image")
        density = round(math.exp(rng.uniform(math.log(low), math.log(high))), 3)
        more = {}
        if op == "options":
            more = {"mode": rng.choice(["sol", "sol", "sol", "exact_only"]), "tokens_first": rng.random() < 0.5,
                    "prepass": rng.random() < 0.5, "diagonal": rng.random() < 0.3, "forced": text > 0}
        c = _case(op, heads, d, block, (frames, rows, cols), density, _beta(kind, max(density, 0.1) if edit else density),
                  batch=batch, text=text, edit=edit, sinks=video, **more)
        n = _tokens(c)
        if op == "host" and batch * heads * n * d > 40 * 32760 * 128:      # pinned memory is slow to make
            continue
        # the smallest: a few thousand tokens over all heads; the largest: the listed one
        if 600 <= n <= 75600 and work(c)["flops"] <= _MOST_FLOPS:
            return c


def _inputs(c, seed):
    """q, k, v [B, H, N, d] as ``synth`` describes them, drawn on the GPU: noise and a shared position feature, sink tokens
    in every frame of a video, the editing target a noisy copy of its source, text tokens without a position."""
    B, H, d, grid = c["batch"], c["heads"], c["d"], (c["frames"], c["rows"], c["cols"])
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    pos = torch.from_numpy(synth.position_features(grid, d)).cuda() * 0.8
    segment = grid[0] * grid[1] * grid[2]
    sink = torch.from_numpy(synth.sink_token_indices(grid)).cuda()
    direction = torch.randn(B, H, 1, d, device="cuda", generator=g)
    out = []
    for name in "qkv":
        x = torch.randn(B, H, segment, d, device="cuda", generator=g) + pos
        if c["sinks"] and name == "q":
            x += 0.1 * direction
        if c["sinks"] and name == "k":
            x[:, :, sink] += 4.0 * direction
        parts = [x.bfloat16()]
        if c["edit"]:
            x += 0.3 * torch.randn(B, H, segment, d, device="cuda", generator=g)
            parts.append(x.bfloat16())
        if c["text"]:
            parts.append(torch.randn(B, H, c["text"], d, device="cuda", generator=g).bfloat16())
        out.append(torch.cat(parts, dim=2) if len(parts) > 1 else parts[0])
    return out


def prepare(case, seed):
    c = case
    q, k, v = _inputs(c, seed)
    B, H, N, d = q.shape
    # sol_attn_dense picks the block size by d
    block = (64 if d == 64 else 128) if c["op"] == "dense" else c["block"]
    ws = sol.make_workspace(B, H, N, d, block, block)
    nq, nk = ws.view.n_q_blocks, ws.view.n_k_blocks
    s = {"op": c["op"], "block": block, "beta": c["beta"], "ws": ws, "shape": (B, H, N, d)}
    if c["op"] == "host":
        s["device"] = [torch.empty_like(q) for _ in range(4)]
        s["host"] = [x.cpu().pin_memory() for x in (q, k, v)] + [torch.empty(q.shape, dtype=q.dtype, pin_memory=True)]
        return s
    if c["op"] == "calibrate":
        sol.sol_attn_bind_workspace(ws)
        sol.sol_attn_pool(q, k, v, block, block, 0.0)
        s["mask"] = torch.zeros(B, H, nq, sol.mask_words(nk), dtype=torch.int32, device="cuda")
        return s
    if c["tokens_first"]:
        q, k, v = (x.transpose(1, 2).contiguous() for x in (q, k, v))
    s.update(q=q, k=k, v=v, out=torch.empty_like(q))
    if c["op"] == "options":
        s["options"] = {"mode": sol.SOL_MODE_EXACT_ONLY if c["mode"] == "exact_only" else sol.SOL_MODE_SOL,
                        "layout": sol.SOL_LAYOUT_BNHD if c["tokens_first"] else sol.SOL_LAYOUT_BHND,
                        "estimator": sol.SOL_EST_DIAGONAL if c["diagonal"] else sol.SOL_EST_MOMENTS}
        if c["prepass"]:
            s["mask"] = torch.zeros(B, H, nq, sol.mask_words(nk), dtype=torch.int32, device="cuda")
            s["options"].update(routing=sol.SOL_ROUTING_PREPASS, mask_out=s["mask"])
        if c["forced"]:                                          # every block that holds a text token
            forced = torch.zeros(nk, dtype=torch.uint8)
            forced[(N - c["text"]) // block:] = 1
            s["options"]["forced_blocks"] = forced.cuda()
    if c["op"] == "topk":
        s["k_blocks"] = max(1, round(c["density"] * nk))
        s["map"] = torch.empty(B, H, nq, nk, device="cuda")
        s["order"] = torch.empty(B, H, nq, nk, dtype=torch.int32, device="cuda")
        s["tau"] = torch.empty(B, H, nq, device="cuda")
    return s


def run(state):
    s = state
    ws, block, beta = s["ws"], s["block"], s["beta"]
    if s["op"] == "options":
        sol.sol_attn_forward_ex(s["q"], s["k"], s["v"], s["out"], ws, block, block, threshold=beta, **s["options"])
        return (s["out"], ws.counts) + ((s["mask"],) if "mask" in s else ())
    sol.sol_attn_bind_workspace(ws)
    if s["op"] == "forward":
        sol.sol_attn_forward(s["q"], s["k"], s["v"], s["out"], block, block, beta)
        return s["out"], ws.counts
    if s["op"] == "dense":
        sol.sol_attn_dense(s["q"], s["k"], s["v"], s["out"])
        return s["out"], ws.counts
    if s["op"] == "host":
        sol.sol_attn_forward_host(*s["host"], *s["device"], block, block, beta)
        return s["host"][3], ws.counts
    if s["op"] == "calibrate":
        sol.sol_attn_thresholds(*s["shape"], block, block, beta)
        sol.sol_attn_route_mask(*s["shape"], block, block, s["mask"])
        return ws.mu, ws.sigma, ws.tau, s["mask"]
    sol.sol_attn_pool(s["q"], s["k"], s["v"], block, block, 0.0)
    sol.sol_attn_route_materialized(ws.qbar, ws.kc, sol.SOL_ROUTE_TOPK, s["k_blocks"], s["map"], s["tau"], order=s["order"])
    sol.sol_attn_forward_ex(s["q"], s["k"], s["v"], s["out"], ws, block, block, skip_pool=True, tau_override=s["tau"])
    return s["out"], ws.counts, s["order"], s["tau"]


def work(case):
    """q, k, v read and the output written once; the products of the selected blocks and of the pooled ones (Eqs. 9-10), at
    the density that the case is meant to have."""
    c = case
    bh, n, d = c["batch"] * c["heads"], _tokens(c), c["d"]
    nb = -(-n // c["block"])
    tensor, pooled = bh * n * d * 2.0, bh * nb * d * 4.0
    proxy = 2.0 * bh * nb * nb * d
    if c["op"] == "calibrate":                                  # pooled queries and keys in, mu, sigma, tau and the bits out
        return {"bytes": 2 * pooled + bh * nb * (12.0 + nb / 8), "flops": 4.0 * bh * nb * d * d + proxy}
    if c["op"] == "dense":
        return {"bytes": 4 * tensor, "flops": 4.0 * bh * n * n * d}
    flops = 4.0 * bh * n * d * (c["density"] * n + (nb if c["mode"] == "sol" else 0)) + proxy
    more = bh * nb * nb * 8.0 if c["op"] == "topk" else 0.0     # the map and the order of its rows
    return {"bytes": 4 * tensor + more, "flops": flops}


def tolerance(case):
    """The outputs are bf16 and P is rounded to bf16: two correct kernels differ by about 2e-3.  A pair of blocks whose score
    meets its threshold to within fp32 rounding may fall on either side (about one in 10^7 pairs does), which changes a count or
    a mask word, and the 128 rows of that query block by as much as one block weighs."""
    if case["op"] == "calibrate":                               # fp32 sums over the pooled keys
        return {"rel": 1e-5, "max": 4e-4, "differ": 1e-4}
    if case["op"] == "dense":
        return {"rel": 8e-3, "max": 0.1}
    return {"rel": 8e-3, "max": 0.9, "differ": 1e-3}


def _softmax_rows(q, k, v, logits_more, v_more, allowed, block):
    """Rows of softmax([q k^T, logits_more]) [v; v_more] where only the key blocks in ``allowed`` [blocks] x rows take part;
    a row without any key is zero."""
    x = q @ k.T
    x.masked_fill_(~allowed.repeat_interleave(block, dim=1)[:, :k.shape[0]], -math.inf)
    if logits_more is not None:
        x, v = torch.cat([x, logits_more], dim=1), torch.cat([v, v_more])
    top = x.amax(dim=1, keepdim=True).clamp_(min=-1e300)
    x.sub_(top).exp_()
    return (x @ v) / x.sum(dim=1, keepdim=True).clamp_(min=1e-300)


def exact(case, seed):
    """What ``run`` returns, from the definitions (Eqs. 3-5 and 9-10) in 64 bits.  Counts, bits and orders have no such value: a
    score within fp32 rounding of its threshold, or of another score, may fall on either side of it."""
    c = case
    n, d = _tokens(c), c["d"]
    if c["op"] != "calibrate" and 4.0 * c["batch"] * c["heads"] * n * n * d > _MOST_FLOPS:
        return None
    q, k, v = (x.flatten(0, 1) for x in _inputs(c, seed))
    block = (64 if d == 64 else 128) if c["op"] == "dense" else c["block"]
    nb, scale = -(-n // block), 1.0 / math.sqrt(d)
    sizes = torch.full((nb, 1), float(block), dtype=torch.float64, device="cuda")
    sizes[-1] = n - (nb - 1) * block

    def pooled(x):
        return torch.nn.functional.pad(x, (0, 0, 0, nb * block - n)).view(nb, block, d).sum(dim=1) / sizes

    forced = torch.zeros(nb, dtype=torch.bool, device="cuda")
    if c["forced"]:
        forced[(n - c["text"]) // block:] = True
    out = torch.empty(q.shape, dtype=torch.float64, device="cuda") if c["op"] != "calibrate" else None
    mus, sigmas, taus = [], [], []
    for h in range(q.shape[0]):
        qh, kh, vh = q[h].double() * scale, k[h].double(), v[h].double()
        qb, kc, vc = pooled(qh), pooled(kh), pooled(vh)
        s = qb @ kc.T
        mu = s.mean(dim=1)
        if c["diagonal"]:
            sigma = (qb.square() @ kc.var(dim=0, correction=0)).sqrt()
        else:
            sigma = s.var(dim=1, correction=0).sqrt()
        tau = mu + c["beta"] * sigma
        if c["op"] == "topk":
            keep = max(1, round(c["density"] * nb))
            ranked = s.sort(dim=1, descending=True).values
            tau = (ranked[:, keep - 1] + ranked[:, keep]) / 2 if keep < nb else torch.full_like(mu, -math.inf)
        mus.append(mu), sigmas.append(sigma), taus.append(tau)
        if out is None:
            continue
        chosen = torch.ones_like(s, dtype=torch.bool) if c["op"] == "dense" else (s > tau[:, None]) | forced
        step = max(1, (1 << 28) // (n * block))                  # query blocks at a time
        for i in range(0, nb, step):
            rows = slice(i * block, min(n, (i + step) * block))
            each = chosen[i:i + step].repeat_interleave(block, dim=0)[:rows.stop - rows.start]
            more = None
            if c["op"] != "dense" and c["mode"] == "sol":
                more = (qh[rows] @ kc.T + sizes.log().T).masked_fill_(each, -math.inf)
            out[h, rows] = _softmax_rows(qh[rows], kh, vh, more, vc, each, block)
    if out is not None:
        out = out.view(c["batch"], c["heads"], n, d)
        out = out.transpose(1, 2).contiguous() if c["tokens_first"] else out
    mu, sigma, tau = (torch.stack(x).view(c["batch"], c["heads"], nb) for x in (mus, sigmas, taus))
    if c["op"] == "calibrate":
        return mu, sigma, tau, None
    if c["op"] == "topk":
        return out, None, None, tau
    return (out, None, None) if c["prepass"] else (out, None)
