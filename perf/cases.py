"""The timed cases: what a user of the package has it do, through its public entry points.

A case names one of six operations:

  layer    ``SubsampledGlobalAttention.forward``: K/V compaction, mean pair and attention of one global block
  frame    ``SubsampledGlobalAttention.frame_attend``: frame attention of a converted early block
  compact  ``SubsampledGlobalAttention.build_kv``: the compaction alone, as a program calls it that shares one
           compact K/V between several attention calls
  project  ``avggt_project_build_kv``: K/V projection with the compaction in its epilogue
  indexed  ``avggt_build_kv_indexed`` + ``avggt_global_attn_indexed``: the layer over a caller-chosen retained set
  host     ``SubsampledGlobalAttention.forward_host``: the layer on pinned host buffers

and the sizes: frames, patch grid, special tokens, heads (of 64), subsampling factor, and the switches.
"""

import math

import torch

import paper_2512_02541_b200 as P
from paper_2512_02541_b200 import binding as B
from paper_2512_02541_b200 import inputs

HEAD_DIM = 64
# the factor's window strides (rows, columns)
STRIDES = {1: (1, 1), 2: (1, 2), 4: (2, 2), 6: (2, 3), 9: (3, 3)}


def _case(name, op, n_frames, sigma, grid_h=37, grid_w=37, n_special=5, n_heads=16, diag=1, mean_fill=2, keep_first=0,
          want_lse=0, recipe="proj", keep=0.0):
    c = dict(op=op, n_frames=n_frames, sigma=sigma, grid_h=grid_h, grid_w=grid_w, n_special=n_special, n_heads=n_heads,
             diag=diag, mean_fill=mean_fill, keep_first=keep_first, want_lse=want_lse, recipe=recipe, keep=keep)
    return c if name is None else dict(name=name, **c)


def listed():
    return [
        # the smallest configuration of the benchmark: four frames of a 16 x 16 grid, independent normal values;
        # a few dozen microseconds, where launches and the latency of a key step count
        _case("tiny_n4_g16_s2", "layer", 4, 2, grid_h=16, grid_w=16, recipe="iid"),
        # ten frames, the shortest sequences the method is used on
        _case("layer_n10_s4", "layer", 10, 4),
        # the VGGT variant (frame 0 uncompressed) on frames that are not square, an odd number of them, with the
        # log-sum-exp that a caller asks for who merges the result with other attention
        _case("layer_n31_s9_first_lse", "layer", 31, 9, grid_h=28, keep_first=1, want_lse=1),
        # the ordinary size: 137,400 queries
        _case("layer_n100_s4", "layer", 100, 4),
        # the benchmark's headline: 1,099,200 queries, where the card runs at its power limit
        _case("layer_n800_s9", "layer", 800, 9),
        # the dense layer, the baseline of every comparison and the first layers of a schedule that keeps them whole
        _case("dense_n100", "layer", 100, 1, diag=0, mean_fill=0),
        # early blocks converted to frame attention, on a short and on an ordinary sequence
        _case("frame_n10", "frame", 10, 4),
        _case("frame_n100", "frame", 100, 4),
        # the compaction on its own at the factor sweep's sequence length
        _case("compact_n333_s4", "compact", 333, 4),
        # the projection that leaves the compact K/V behind, with the full K and V written for the diagonal
        _case("project_n100_s4", "project", 100, 4),
        # a caller's own selection (a random fifth of the patches, as in the comparison of selectors)
        _case("indexed_n57", "indexed", 57, 4, grid_h=28, keep=0.2),
        # the layer end to end from host memory, copies included
        _case("host_n100_s4", "host", 100, 4),
    ]


# the ranges that draw() covers: operation, its share, most frames
_OPS = (("layer", 0.5, 360), ("frame", 0.16, 360), ("compact", 0.12, 500), ("project", 0.12, 300), ("indexed", 0.07, 150),
        ("host", 0.03, 60))
# patch grids: square frames, the tests' sizes, and the non-square frames of patch-14 images
_GRIDS = ((37, 37), (37, 37), (37, 37), (28, 37), (37, 28), (16, 16), (21, 37), (12, 13), (24, 31))
_MAX_FLOPS = 2.0e14   # a third of the largest listed case


def draw(rng):
    x = rng.random()
    for op, share, most in _OPS:
        if x < share:
            break
        x -= share
    grid_h, grid_w = rng.choice(_GRIDS)
    n_frames = int(round(math.exp(rng.uniform(0.0, math.log(most)))))
    sigma = rng.choice((1, 2, 4, 4, 6, 6, 9, 9))
    dense = sigma == 1
    c = _case(None, op, n_frames, sigma, grid_h=grid_h, grid_w=grid_w, n_special=rng.choice((5, 5, 5, 1, 0)),
              n_heads=rng.choice((16, 16, 16, 12, 8, 6)), diag=0 if dense else rng.choice((1, 1, 1, 0)),
              mean_fill=0 if dense else rng.choice((2, 2, 2, 1, 0)), keep_first=rng.choice((0, 0, 1)),
              want_lse=rng.choice((0, 0, 0, 1)) if op in ("layer", "frame", "indexed") else 0,
              keep=round(rng.uniform(0.05, 0.5), 3) if op == "indexed" else 0.0)
    while work(c)["flops"] > _MAX_FLOPS:
        c["n_frames"] = max(1, int(c["n_frames"] * 0.8))
    return c


def _tokens(c):
    """(tokens per frame, tokens, retained tokens)"""
    L = c["n_special"] + c["grid_h"] * c["grid_w"]
    n_tok = c["n_frames"] * L
    if c["op"] == "indexed":
        patches = c["n_frames"] * c["grid_h"] * c["grid_w"]
        return L, n_tok, c["n_frames"] * c["n_special"] + max(1, int(patches * c["keep"]))
    sh, sw = STRIDES[c["sigma"]]
    Lc = c["n_special"] + -(-c["grid_h"] // sh) * -(-c["grid_w"] // sw)
    return L, n_tok, c["n_frames"] * Lc + (L - Lc if c["keep_first"] else 0)


def work(case):
    c = case
    L, n_tok, M = _tokens(c)
    C = c["n_heads"] * HEAD_DIM
    row = 2 * C                                   # bytes of one token's row of Q, K, V or O
    lse = 4 * n_tok * c["n_heads"] if c["want_lse"] else 0
    has_mean = c["mean_fill"] != 0 and M < n_tok
    if c["op"] == "frame":
        return {"bytes": 4 * n_tok * row + lse, "flops": 4.0 * n_tok * L * C}
    if c["op"] == "compact":
        read = n_tok if has_mean else M
        return {"bytes": 2 * (read + M) * row + 4 * M + 8 * C * has_mean, "flops": 2.0 * (n_tok - M) * C * has_mean}
    if c["op"] == "project":
        # X and both weights read; K, V, Kc, Vc and the index list written
        return {"bytes": n_tok * row + 2 * C * row + 2 * (n_tok + M) * row + 4 * M, "flops": 4.0 * n_tok * C * C}
    extra = (1 if c["diag"] else 0) + (1 if has_mean else 0)
    kv = n_tok if has_mean or c["diag"] else M    # rows of K and V that matter
    return {"bytes": 2 * n_tok * row + 2 * kv * row + lse + (4 * M if c["op"] == "indexed" else 0),
            "flops": 4.0 * n_tok * (M + extra) * C}


def tolerance(case):
    # about four times what the paths were seen to differ by from 64-bit sums whose results are rounded to the same types
    if case["op"] == "compact":
        return {"rel": 5e-7, "max": 1e-6}         # copies, and 32-bit sums over the dropped rows (seen: 7e-8, 2e-7)
    if case["op"] == "project":
        return {"rel": 3e-4, "max": 3e-2}         # bf16 results of 32-bit sums: a last bit now and then (seen: 6e-5, 8e-3)
    return {"rel": 7e-3, "max": 4e-2}             # sums with weights rounded to bf16 (seen: 1.8e-3, 1.2e-2)


def _params(c):
    return P.make_params(c["n_frames"], c["grid_h"], c["grid_w"], c["n_special"], c["n_heads"], HEAD_DIM, c["sigma"],
                         diag=c["diag"], mean_fill=c["mean_fill"], keep_first_frame=bool(c["keep_first"]))


def prepare(case, seed):
    c = case
    wl = inputs.Workload("case", c["n_frames"], c["grid_h"], c["grid_w"], c["n_special"], c["n_heads"], HEAD_DIM, c["sigma"],
                         c["diag"], c["mean_fill"], c["recipe"], c["keep_first"])
    params = _params(c)
    L, n_tok, M = _tokens(c)
    H, C = c["n_heads"], c["n_heads"] * HEAD_DIM
    dev = "cuda"
    s = {"op": c["op"], "params": params}
    if c["op"] == "project":
        gen = torch.Generator(device=dev)
        gen.manual_seed(seed)
        normal = lambda *shape: torch.randn(shape, generator=gen, device=dev, dtype=torch.float32)
        s["C"] = C
        s["X"] = normal(n_tok, C).bfloat16()
        s["Wk"], s["Wv"] = (normal(C, C) * C ** -0.5).bfloat16(), (normal(C, C) * C ** -0.5).bfloat16()
        s["bk"], s["bv"] = normal(C), normal(C)
        s["K"], s["V"] = (torch.empty((n_tok, H, HEAD_DIM), dtype=torch.bfloat16, device=dev) for _ in range(2))
        s["Kc"], s["Vc"] = (torch.empty((H, M, HEAD_DIM), dtype=torch.bfloat16, device=dev) for _ in range(2))
        s["idx"] = torch.empty((M,), dtype=torch.int32, device=dev)
        s["kmean"], s["vmean"] = (torch.zeros((H, HEAD_DIM), dtype=torch.float32, device=dev) for _ in range(2))
        s["ws"] = torch.empty((B.avggt_project_workspace_bytes(params, C),), dtype=torch.uint8, device=dev)
        return s
    Q, K, V = inputs.make_qkv(wl, seed=seed, device=dev)
    if c["op"] == "indexed":
        gen = torch.Generator(device=dev)
        gen.manual_seed(seed + 1)
        tok = torch.arange(n_tok, device=dev)
        special = tok[tok % L < c["n_special"]]
        patch = tok[tok % L >= c["n_special"]]
        picked = patch[torch.randperm(patch.numel(), generator=gen, device=dev)[:M - special.numel()]]
        s["idx"] = torch.sort(torch.cat([special, picked])).values.to(torch.int32)
        s["M"] = M
        s["Q"], s["K"], s["V"] = Q, K, V
        s["Kc"], s["Vc"] = (torch.empty((H, M, HEAD_DIM), dtype=torch.bfloat16, device=dev) for _ in range(2))
        s["slots"] = torch.empty((n_tok,), dtype=torch.int32, device=dev)
        s["kmean"], s["vmean"] = (torch.zeros((H, HEAD_DIM), dtype=torch.float32, device=dev) for _ in range(2))
        build_ws, attn_ws = B.avggt_workspace_bytes(params)
        s["build_ws"] = torch.empty((max(build_ws, 16),), dtype=torch.uint8, device=dev)
        s["attn_ws"] = torch.zeros((max(attn_ws, 16),), dtype=torch.uint8, device=dev)
        s["lse"] = torch.empty((n_tok, H), dtype=torch.float32, device=dev) if c["want_lse"] else None
        return s
    s["layer"] = P.SubsampledGlobalAttention(params, device=dev, want_lse=bool(c["want_lse"]))
    if c["op"] == "host":
        pinned = lambda: torch.empty((n_tok, H, HEAD_DIM), dtype=torch.bfloat16, pin_memory=True)
        for name, t in (("Q", Q), ("K", K), ("V", V)):
            s[name] = pinned()
            s[name].copy_(t)
        s["O"] = pinned()
        return s
    s["Q"], s["K"], s["V"] = Q, K, V
    return s


def run(state):
    s = state
    op = s["op"]
    if op == "layer":
        layer = s["layer"]
        O = layer.forward(s["Q"], s["K"], s["V"])
        return O if layer.lse is None else (O, layer.lse)
    if op == "frame":
        layer = s["layer"]
        O = layer.frame_attend(s["Q"], s["K"], s["V"])
        return O if layer.lse is None else (O, layer.lse)
    if op == "compact":
        layer = s["layer"]
        layer.build_kv(s["K"], s["V"])
        return layer.Kc, layer.Vc, layer.idx, layer.kmean, layer.vmean
    if op == "host":
        return s["layer"].forward_host(s["Q"], s["K"], s["V"], s["O"])
    stream = torch.cuda.current_stream().cuda_stream
    if op == "project":
        B.avggt_project_build_kv(s["params"], s["C"], s["X"], s["Wk"], s["Wv"], s["bk"], s["bv"], s["K"], s["V"], s["Kc"],
                                 s["Vc"], s["idx"], s["kmean"], s["vmean"], s["ws"], s["ws"].numel(), stream)
        return s["K"], s["V"], s["Kc"], s["Vc"], s["idx"], s["kmean"], s["vmean"]
    O = torch.empty_like(s["Q"])
    B.avggt_build_kv_indexed(s["params"], s["idx"], s["M"], s["K"], s["V"], s["Kc"], s["Vc"], s["slots"], s["kmean"],
                             s["vmean"], s["build_ws"], s["build_ws"].numel(), stream)
    B.avggt_global_attn_indexed(s["params"], s["M"], s["slots"], s["Q"], s["K"], s["V"], s["Kc"], s["Vc"], s["kmean"],
                                s["vmean"], O, s["lse"], s["attn_ws"], s["attn_ws"].numel(), stream)
    return O if s["lse"] is None else (O, s["lse"])
