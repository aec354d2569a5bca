"""Calls that follow one another without a wait, where a kernel begins while the one that writes its input still runs: each reads
what was written, not what was there before."""

import pytest
import torch

import paper_2512_02541_b200 as P
from paper_2512_02541_b200 import inputs

pytestmark = pytest.mark.gpu


# 1,485 tokens: one cluster per head; 12,045: a warp per row (the limit is 5,760 at 16 heads)
@pytest.mark.parametrize("n_frames", (9, 73))
def test_retained_sets_in_turn(n_frames):
    wl = inputs.Workload("turns", n_frames, 16, 10, 5, 16, 64, 4, 1, 2, "iid")
    params = P.make_params(wl.n_frames, wl.grid_h, wl.grid_w, wl.n_special, wl.n_heads, wl.head_dim, wl.sigma)
    _, K, V = inputs.make_qkv(wl, seed=1, device="cuda")
    H, d, n_tok = wl.n_heads, wl.head_dim, wl.n_tokens
    gen = torch.Generator(device="cuda").manual_seed(7)
    M = n_tok // 3
    lists = [torch.sort(torch.randperm(n_tok, generator=gen, device="cuda")[:M]).values.to(torch.int32) for _ in range(2)]
    calls = 40
    Kc = torch.full((calls, H, M, d), float("nan"), dtype=torch.bfloat16, device="cuda")
    Vc = torch.full_like(Kc, float("nan"))
    means = torch.full((calls, 2, H, d), float("nan"), device="cuda")
    idx = torch.empty_like(lists[0])                                      # one list and one map, written again for every call
    slots = torch.empty((n_tok,), dtype=torch.int32, device="cuda")
    ws = torch.empty((P.avggt_workspace_bytes(params)[0],), dtype=torch.uint8, device="cuda")
    for c in range(calls):
        idx.copy_(lists[c & 1])
        P.avggt_build_kv_indexed(params, idx, M, K, V, Kc[c], Vc[c], slots, means[c, 0], means[c, 1], ws, ws.numel())
    torch.cuda.synchronize()
    for which in range(2):
        rows = lists[which].long()
        dropped = torch.ones(n_tok, dtype=torch.bool, device="cuda")
        dropped[rows] = False
        for c in range(which, calls, 2):
            assert torch.equal(Kc[c], K[rows].transpose(0, 1)) and torch.equal(Vc[c], V[rows].transpose(0, 1)), c
            for got, src in ((means[c, 0], K), (means[c, 1], V)):         # 32-bit sums of values around 1: 1e-5 of them, as elsewhere
                assert (got.double() - src[dropped].double().mean(0)).abs().max() <= 1e-5, c


@pytest.mark.parametrize("n_frames,mean_fill", [(9, 2), (73, 2), (73, 0)])
def test_compaction_of_what_the_projection_has_just_written(n_frames, mean_fill):
    wl = inputs.Workload("projected", n_frames, 16, 10, 5, 16, 64, 4, 1, mean_fill, "iid")
    params = P.make_params(wl.n_frames, wl.grid_h, wl.grid_w, wl.n_special, wl.n_heads, wl.head_dim, wl.sigma, mean_fill=mean_fill)
    H, d, n_tok, C = wl.n_heads, wl.head_dim, wl.n_tokens, 256
    gen = torch.Generator(device="cuda").manual_seed(8)
    normal = lambda *shape: torch.randn(shape, generator=gen, device="cuda").bfloat16()
    X, W = [normal(n_tok, C) for _ in range(2)], normal(H * d, C)
    K, V = (torch.empty((n_tok, H, d), dtype=torch.bfloat16, device="cuda") for _ in range(2))
    M, _ = P.avggt_kv_count(params)
    pairs = torch.full((8, 2, 2, H, M, d), float("nan"), dtype=torch.bfloat16, device="cuda")   # call, projection or compaction, K or V
    layer = P.SubsampledGlobalAttention(params)
    ws = torch.empty((P.avggt_project_workspace_bytes(params, C),), dtype=torch.uint8, device="cuda")
    for c in range(pairs.shape[0]):
        P.avggt_project_build_kv(params, C, X[c & 1], W, W, None, None, K, V, pairs[c, 0, 0], pairs[c, 0, 1], None, layer.kmean,
                                 layer.vmean, ws, ws.numel())
        P.avggt_build_kv(params, K, V, pairs[c, 1, 0], pairs[c, 1, 1], None, layer.kmean, layer.vmean, layer.build_ws,
                         layer.build_ws.numel())
    torch.cuda.synchronize()
    P.avggt_check_status(ws)
    assert torch.isfinite(pairs.float()).all()
    assert torch.equal(pairs[:, 0], pairs[:, 1])
    assert torch.equal(pairs[0], pairs[2]) and not torch.equal(pairs[0], pairs[1])
