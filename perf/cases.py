"""The work whose speed is measured: whole requests of block-wise prefill under a KV budget.

A pass takes one request through the library as a program that serves such requests does: the caches of all layers are
reset, every block of the prefix goes through every layer, and the request ends with compressed caches and the attention
output of every token.  Inputs are shaped like the workloads of ``paper_2604_16734_b200.workloads`` (an image, a tiled
image, a video; patches first, the text prompt last).

A case is a dict:

  kind, grid_h, grid_w, units, text     the prefix: ``units`` tiles or frames of grid_h x grid_w patches, then text tokens
  layers, hq, hkv, d, dtype             the attention shape
  chunk, budget                         tokens per block, entries kept per (layer, kv-head)
  policy                                "attn" (query-aware score) or "keydiff" (query-agnostic)
  proxy                                 proxy query tokens that ride along with every vision block (0: none)
  hybrid                                the first ``budget`` tokens go through in one pass
  overlap                               score / select / compact of a layer beside the next layer's attention
  how                                   "calls" one call per (block, layer); "graph" those calls replayed from a CUDA
                                        graph; "host" inputs and outputs in pinned host memory
"""
import math

import torch

from paper_2604_16734_b200.binding import KVC_FLAG_ASYNC_COMPRESS, KVC_SCORE_ATTN, KVC_SCORE_KEYDIFF, Kvc
from paper_2604_16734_b200.workloads import Workload, WorkloadConfig

WINDOW = 32          # observer rows per block (the library's default)


def _case(name, kind, grid, units, text, layers, heads, d, chunk, budget, dtype="bf16", policy="attn", proxy=0,
          hybrid=False, overlap=False, how="calls"):
    c = dict(kind=kind, grid_h=grid[0], grid_w=grid[1], units=units, text=text, layers=layers, hq=heads[0], hkv=heads[1],
             d=d, dtype=dtype, chunk=chunk, budget=budget, policy=policy, proxy=proxy, hybrid=hybrid, overlap=overlap, how=how)
    return dict(name=name, **c) if name else c


def listed():
    return [
        # The smallest request: a thumbnail with a short question, two layers, every size odd.  Latency and launches.
        _case("thumbnail", "image", (7, 9), 1, 17, 2, (8, 2), 64, 32, 48),
        # fp32, for programs that check or calibrate at full precision: one image through one layer (the repository's
        # smallest configuration) ...
        _case("image_fp32", "image", (24, 24), 1, 32, 1, (4, 1), 64, 64, 128, dtype="fp32"),
        # ... and a tiled image with larger blocks and grouped heads.
        _case("tiles_fp32", "tiles", (24, 24), 3, 57, 2, (8, 2), 128, 576, 512, dtype="fp32"),
        # One image for a model with as many kv-heads as query heads: the calls one by one, in stream order (the
        # library's defaults), and the same request served from a captured graph with overlapped compression.
        _case("image", "image", (24, 24), 1, 64, 32, (32, 32), 128, 128, 192),
        _case("image_graph", "image", (24, 24), 1, 64, 32, (32, 32), 128, 128, 192, overlap=True, how="graph"),
        # A high-resolution image in tiles, seven query heads per kv-head, one tile per block.
        _case("tiles_graph", "tiles", (24, 24), 5, 128, 28, (28, 4), 128, 576, 1024, overlap=True, how="graph"),
        # Larger tiles in the default block size of 256 with the prompt's first tokens as observers of every block.
        _case("tiles_proxy", "tiles", (28, 28), 6, 128, 4, (28, 4), 128, 256, 2048, proxy=32),
        # A video, one frame per block (196 tokens: no multiple of a tile).
        _case("video_graph", "video", (14, 14), 64, 128, 8, (32, 8), 128, 196, 2048, overlap=True, how="graph"),
        # The query-agnostic policy, calls one by one in stream order, head dimension 64, ragged blocks.
        _case("video_keydiff", "video", (13, 15), 24, 51, 6, (16, 4), 64, 333, 1500, policy="keydiff"),
        # Long video: the largest request, large blocks and budget.
        _case("long_video_graph", "video", (12, 12), 256, 256, 4, (32, 8), 128, 1024, 4096, overlap=True, how="graph"),
        # The same kind of request in stream order, the first 4096 tokens in one pass.
        _case("long_video_hybrid", "video", (12, 12), 128, 256, 2, (32, 8), 128, 1024, 4096, hybrid=True),
        # A program whose activations live in host memory.
        _case("video_host", "video", (14, 14), 16, 128, 3, (32, 8), 128, 196, 1024, how="host"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    most = {"bf16": max(work(c)["flops"] for c in listed()), "fp32": max(work(c)["flops"] for c in listed() if c["dtype"] == "fp32")}
    while True:
        kind = rng.choice(["image", "tiles", "video"])
        dtype = "fp32" if rng.random() < 0.2 else "bf16"
        hi = {"image": 36, "tiles": 28, "video": 16}[kind]
        grid = (rng.randint(7, hi), rng.randint(7, hi))
        units = {"image": 1, "tiles": _log(rng, 2, 10), "video": _log(rng, 8, 200)}[kind]
        d = rng.choice([64, 128, 128])
        heads = rng.choice([(4, 1), (8, 2), (8, 8), (12, 4), (16, 4), (28, 4), (32, 8), (32, 32)])
        chunk = grid[0] * grid[1] if rng.random() < 0.4 else _log(rng, 32, 1024)
        budget = _log(rng, 48, 4096)
        policy = "keydiff" if rng.random() < 0.2 else "attn"
        proxy = rng.choice([8, 16, 32]) if policy == "attn" and rng.random() < 0.25 else 0
        hybrid = not proxy and rng.random() < 0.25
        how = rng.choice(["calls", "calls", "graph", "graph", "host"])
        overlap = how != "host" and dtype == "bf16" and rng.random() < 0.5
        c = _case(None, kind, grid, units, max(_log(rng, 8, 256), proxy), _log(rng, 1, 32), heads, d, chunk, budget, dtype,
                  policy, proxy, hybrid, overlap, how)
        tokens = grid[0] * grid[1] * units
        calls = len(_calls(c)) * c["layers"]
        elems = sum(x[1] for x in _calls(c)) * c["layers"] * 2 * (heads[0] + heads[1]) * d
        host = 120e6 if how == "host" else 1.6e9
        if tokens > budget and calls <= 1200 and elems <= host and work(c)["flops"] <= most[dtype]:
            return c


def _config(case):
    return WorkloadConfig("request", 7, case["layers"], case["hq"], case["hkv"], case["d"], case["dtype"],
                          (case["grid_h"], case["grid_w"]), case["units"], case["text"], case["chunk"], case["budget"],
                          case["kind"], rho=0.95, scene_cut=32, shared_rank=8, mix_layers=False, obs_window=WINDOW)


def _calls(case):
    """(first row in the packed inputs, rows, proxy rows among them, position of the first token) of every block."""
    cfg = _config(case)
    out, row = [], 0
    for pos, n in (cfg.chunks_hybrid() if case["hybrid"] else cfg.chunks()):
        t = case["proxy"] if pos < cfg.n_vision else 0
        out.append((row, n + t, t, pos))
        row += n + t
    return out


def prepare(case, seed):
    cfg, calls = _config(case), _calls(case)
    wl = Workload(cfg, device="cuda", seed=seed)
    index = None
    if case["proxy"]:          # a block's proxies follow it in the packed inputs
        index = torch.cat([torch.cat([torch.arange(p, p + n - t), torch.arange(cfg.n_vision, cfg.n_vision + t)])
                           for _, n, t, p in calls]).cuda()
    layers = []
    for i in range(cfg.n_layers):
        qkv = wl.layer(i)
        layers.append([x if index is None else x[index].contiguous() for x in qkv])
    outs = [torch.zeros_like(q) for q, _, _ in layers]
    if case["how"] == "host":
        layers = [[x.cpu().pin_memory() for x in qkv] for qkv in layers]
        outs = [x.cpu().pin_memory() for x in outs]
    kvc = Kvc(cfg.n_layers, cfg.n_q_heads, cfg.n_kv_heads, cfg.head_dim, cfg.torch_dtype, cfg.budget,
              cfg.chunk + case["proxy"], cfg.obs_window, flags=KVC_FLAG_ASYNC_COMPRESS if case["overlap"] else 0,
              policy=KVC_SCORE_KEYDIFF if case["policy"] == "keydiff" else KVC_SCORE_ATTN)
    steps = [(i, *(x[row:row + n] for x in layers[i]), t, pos, outs[i][row:row + n])
             for row, n, t, pos in calls for i in range(cfg.n_layers)]
    left = min(cfg.budget, cfg.n_tokens)
    state = dict(kvc=kvc, how=case["how"], overlap=case["overlap"], steps=steps, outs=outs, inputs=layers,
                 cached=[kvc.cache_view(i)[2][:, :left] for i in range(cfg.n_layers)], tokens=cfg.n_tokens, graph=None)
    if case["how"] == "graph":
        _request(state)
        torch.cuda.synchronize()
        state["graph"] = torch.cuda.CUDAGraph()
        with torch.cuda.graph(state["graph"]):
            state["result"] = _request(state)
    return state


def _request(state):
    """One request.  Returns the attention outputs and, per layer and kv-head, which tokens the cache still holds (the
    order of a cache's entries is unspecified)."""
    kvc = state["kvc"]
    kvc.reset()
    for layer, q, k, v, proxy, pos, out in state["steps"]:
        if state["how"] == "host":
            kvc.prefill_chunk_host(layer, q, k, v, pos, out)
        elif proxy:
            kvc.prefill_chunk_proxy(layer, q, k, v, proxy, pos, out)
        else:
            kvc.prefill_chunk(layer, q, k, v, pos, out)
    if state["how"] == "host":
        kvc.host_flush()
    if state["overlap"]:
        kvc.join()
    pos = torch.stack(state["cached"])
    held = torch.zeros(pos.shape[0], pos.shape[1], state["tokens"], dtype=torch.bool, device=pos.device)
    held.scatter_(2, pos.long(), True)
    return {"out": state["outs"], "held": held}


def run(state):
    if state["graph"] is not None:
        state["graph"].replay()
        return state["result"]
    return _request(state)


def work(case):
    """Per block and layer: q, k, v and the cached keys and values read, the output and the new entries written; the two
    contractions of the attention and the observers' scores."""
    hq, hkv, d, size = case["hq"], case["hkv"], case["d"], 4 if case["dtype"] == "fp32" else 2
    held, moved, flops = 0, 0, 0
    for _, n, t, _ in _calls(case):
        moved += size * d * (2 * n * hq + 2 * n * hkv + 2 * (n - t) * hkv + 2 * held * hkv)
        flops += 4 * hq * d * (n * held + n * (n + 1) // 2)
        total = held + n - t
        if total > case["budget"]:
            flops += 2 * hkv * d * total * 2 if case["policy"] == "keydiff" else 2 * hq * d * (t or min(WINDOW, n)) * total
        held = min(total, case["budget"])
    return {"bytes": moved * case["layers"], "flops": flops * case["layers"]}


def tolerance(case):
    # Measured over the listed and eight drawn cases.  fp32: against a double-precision run of the method, rel up to
    # 4.3e-7 and max up to 5.5e-6.  bf16: with the key range split differently, and with probabilities kept in fp32
    # (the library's CUDA-core kernels), rel up to 1.44e-3 and max up to 1.3e-2.  About four times that is allowed.  No
    # retained set differed in any of these runs; the share allowed is for near-ties at the cut-off.
    if case["dtype"] == "fp32":
        return {"rel": 2e-6, "max": 2.2e-5, "differ": 5e-4}
    return {"rel": 6e-3, "max": 5e-2, "differ": 5e-4}
