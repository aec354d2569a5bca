"""The compaction kernels (few tokens: a cluster of thread blocks per head; many, with a mean: tiles of tokens; without: tiles of compact
rows) over the head counts that select their variants, against the oracle: bit copies, indices, and the mean pair."""

import pytest
import torch

import paper_2512_02541_b200 as P
from paper_2512_02541_b200 import inputs

from test_gpu_parity import _cfgs, _check_build

pytestmark = pytest.mark.gpu


# 16 to 1 groups of adding threads and one or two chunks per thread in the many-token kernel, tiles of 4 to 32 rows; clusters of 8, 4, 2
# blocks in the few-token kernel, whose limit lies at 8,800 tokens for up to 6 heads, 4,400 up to 18, 2,200 above; 12,300 and 1,230 tokens,
# not a multiple of any group
@pytest.mark.parametrize("heads", (1, 3, 6, 7, 8, 12, 16, 19, 24, 28, 32))
@pytest.mark.parametrize("n_frames", (3, 30))
@pytest.mark.parametrize("mean_fill,keep_first", [(2, 1), (0, 0)])
def test_compaction(heads, n_frames, mean_fill, keep_first):
    wl = inputs.Workload("compaction", n_frames, 15, 27, 5, heads, 64, 6, 1, mean_fill, "iid", keep_first_frame=keep_first)
    params, ocfg = _cfgs(wl)
    _, K, V = inputs.make_qkv(wl, seed=heads, device="cuda")
    layer = P.SubsampledGlobalAttention(params)
    for t in (layer.Kc, layer.Vc, layer.kmean, layer.vmean):
        t.fill_(float("nan"))
    layer.idx.fill_(-1)
    layer.build_kv(K, V)
    torch.cuda.synchronize()
    _check_build(ocfg, layer, K, V)


# both kernels with nothing to average: the mean pair is zero-filled, as the first part of the layer writes it and as a shard's sums
@pytest.mark.parametrize("n_frames", (3, 30))
def test_nothing_dropped(n_frames):
    wl = inputs.Workload("whole", n_frames, 15, 27, 5, 16, 64, 1, 1, 2, "iid")
    params, ocfg = _cfgs(wl)
    _, K, V = inputs.make_qkv(wl, seed=1, device="cuda")
    layer = P.SubsampledGlobalAttention(params)
    for t in (layer.kmean, layer.vmean):
        t.fill_(float("nan"))
    layer.build_kv(K, V)
    slot_rows = layer.M + 3
    slot = torch.full((2, wl.n_heads, slot_rows, 64), float("nan"), dtype=torch.bfloat16, device="cuda")
    sums = torch.full((2, wl.n_heads, 64), float("nan"), device="cuda")
    P.avggt_build_kv_shard(params, K, V, slot, slot_rows, None, sums, layer.build_ws, layer.build_ws.numel())
    torch.cuda.synchronize()
    _check_build(ocfg, layer, K, V)
    assert not layer.kmean.any() and not layer.vmean.any() and not sums.any()
    assert torch.equal(slot[0, :, :layer.M], layer.Kc) and torch.equal(slot[1, :, :layer.M], layer.Vc)
    assert torch.isnan(slot[:, :, layer.M:].float()).all()


# Tiles of 8 tokens (16 heads) or 4 (32), 296 blocks, three tiles in flight in each: token counts around a tile, around the tiles of all
# blocks together, and around the ring; with a mean and, over the compact rows (tiles of 6 of 24 heads, of 5 of 32, 148 blocks), without
@pytest.mark.parametrize("heads,n_tok", [(16, t) for t in (4401, 4409, 4736 * 8 - 1, 7104, 7105, 7111)] + [(32, 2201), (32, 3 * 1184 + 5)]
                         + [(24, t) for t in (2663, 2664, 2665)] + [(32, 2221)])
@pytest.mark.parametrize("sigma,mean_fill", [(4, 2), (4, 0), (1, 2)])
def test_tokens_around_a_tile(heads, n_tok, sigma, mean_fill):
    wl = inputs.Workload("tiles", 1, 3, (n_tok - 2) // 3, 2 + (n_tok - 2) % 3, heads, 64, sigma, 1, mean_fill, "iid")
    assert wl.n_tokens == n_tok
    params, ocfg = _cfgs(wl)
    _, K, V = inputs.make_qkv(wl, seed=n_tok, device="cuda")
    layer = P.SubsampledGlobalAttention(params)
    for t in (layer.Kc, layer.Vc, layer.kmean, layer.vmean):
        t.fill_(float("nan"))
    layer.idx.fill_(-1)
    layer.build_kv(K, V)
    torch.cuda.synchronize()
    _check_build(ocfg, layer, K, V)


def test_a_list_with_entries_that_are_no_token():
    """Their compact rows are left as they were; without a mean the list itself says what is read."""
    wl = inputs.Workload("listed", 4, 37, 37, 5, 16, 64, 4, 1, 0, "iid")
    params, _ = _cfgs(wl)
    _, K, V = inputs.make_qkv(wl, seed=1, device="cuda")
    for n_kept in (5, 64, 701):
        idx = torch.sort(torch.randperm(wl.n_tokens, device="cuda")[:n_kept]).values.to(torch.int32)
        idx[-1] = wl.n_tokens + 3
        idx[0] = -1
        Kc, Vc = (torch.full((wl.n_heads, n_kept, 64), 7.0, dtype=torch.bfloat16, device="cuda") for _ in range(2))
        slots = torch.empty((wl.n_tokens,), dtype=torch.int32, device="cuda")
        ws = torch.empty((P.avggt_workspace_bytes(params)[0],), dtype=torch.uint8, device="cuda")
        P.avggt_build_kv_indexed(params, idx, n_kept, K, V, Kc, Vc, slots, None, None, ws, ws.numel())
        torch.cuda.synchronize()
        kept = idx[1:-1].long()
        for full, compact in ((K, Kc), (V, Vc)):
            assert torch.equal(compact[:, 1:-1], full[kept].transpose(0, 1))
            assert (compact[:, 0] == 7).all() and (compact[:, -1] == 7).all()


# on either side of the few-token limit of 16 heads (4,400 tokens), with a mean and without
@pytest.mark.parametrize("n_frames", (3, 4))
@pytest.mark.parametrize("mean_fill", (0, 2))
def test_a_list_with_a_repeated_entry(n_frames, mean_fill):
    """One of its two compact rows, the one that the map names, is written."""
    wl = inputs.Workload("repeated", n_frames, 37, 37, 5, 16, 64, 4, 1, mean_fill, "iid")
    params, _ = _cfgs(wl)
    _, K, V = inputs.make_qkv(wl, seed=1, device="cuda")
    n_kept = 300
    idx = torch.sort(torch.randperm(wl.n_tokens, device="cuda")[:n_kept]).values.to(torch.int32)
    for m in (1, 9, 100, n_kept - 1):   # within a tile of eight, across two, at the end
        idx[m] = idx[m - 1]
    Kc, Vc = (torch.full((wl.n_heads, n_kept, 64), 7.0, dtype=torch.bfloat16, device="cuda") for _ in range(2))
    slots = torch.empty((wl.n_tokens,), dtype=torch.int32, device="cuda")
    kmean, vmean = (torch.zeros((wl.n_heads, 64), device="cuda") for _ in range(2))
    ws = torch.empty((P.avggt_workspace_bytes(params)[0],), dtype=torch.uint8, device="cuda")
    P.avggt_build_kv_indexed(params, idx, n_kept, K, V, Kc, Vc, slots, kmean, vmean, ws, ws.numel())
    torch.cuda.synchronize()
    named = slots[idx.long()] == torch.arange(n_kept, dtype=torch.int32, device="cuda")
    assert int((~named).sum()) == 4
    for full, compact in ((K, Kc), (V, Vc)):
        assert torch.equal(compact[:, named], full[idx.long()[named]].transpose(0, 1))
        assert (compact[:, ~named] == 7).all()


def test_a_workspace_for_a_block_per_sm():
    """Above 16 heads a call gets by with half of what avggt_workspace_bytes asks for, on half as many blocks."""
    wl = inputs.Workload("half", 6, 37, 37, 5, 20, 64, 4, 1, 2, "iid")
    params, ocfg = _cfgs(wl)
    _, K, V = inputs.make_qkv(wl, seed=2, device="cuda")
    layer = P.SubsampledGlobalAttention(params)
    half = torch.cuda.get_device_properties(0).multi_processor_count * 2 * 20 * 64 * 4
    assert half < layer.build_ws_bytes
    ws = torch.empty((half,), dtype=torch.uint8, device="cuda")
    P.avggt_build_kv(params, K, V, layer.Kc, layer.Vc, layer.idx, layer.kmean, layer.vmean, ws, half)
    torch.cuda.synchronize()
    _check_build(ocfg, layer, K, V)
    with pytest.raises(P.AvggtError):
        P.avggt_build_kv(params, K, V, layer.Kc, layer.Vc, layer.idx, layer.kmean, layer.vmean, ws, half - 1)


def test_a_tensor_map_that_cannot_be_encoded_is_named():
    """Tensor maps have strides below 2^40 bytes; a slot of more rows than that is refused before anything is launched."""
    wl = inputs.Workload("stride", 6, 37, 37, 5, 16, 64, 4, 1, 2, "iid")
    params, _ = _cfgs(wl)
    _, K, V = inputs.make_qkv(wl, seed=3, device="cuda")
    layer = P.SubsampledGlobalAttention(params)
    sums = torch.zeros((2, wl.n_heads, 64), device="cuda")
    for p in (params, P.make_params(6, 37, 37, 5, 16, 64, 4, diag=0, mean_fill=0)):
        with pytest.raises(P.AvggtError, match="cuTensorMapEncodeTiled"):
            P.avggt_build_kv_shard(p, K, V, layer.Kc, 1 << 34, None, sums, layer.build_ws, layer.build_ws.numel())
    torch.cuda.synchronize()
    assert not sums.any()
