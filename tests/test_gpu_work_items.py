"""How the attention kernel cuts a launch: full items (256 rows), half items where the chip has room for all of them, a last
item whose rows are spread over both tiles, several items per thread block, key counts around the 112-key step; and the
one-call layer against its two calls."""

import numpy as np
import pytest
import torch

import paper_2512_02541_b200 as P
from paper_2512_02541_b200 import binding as B
from paper_2512_02541_b200 import inputs, sharded

import test_gpu_frame_attn as frame_attn
import test_gpu_indexed as indexed
from test_gpu_parity import _check_attn, _host, _run_gpu

pytestmark = pytest.mark.gpu


# 32 heads: 769 to 1,023 queries make one round of 256-row items, 1,281 two rounds of 160- or 144-row ones, 2,305 three rounds (several
# items per thread block); the last item has 1, 16, 17, 128, 129 or 255 rows of 256.  4 heads: items of 128 rows, or of 256 with
# nothing dropped and up to 129 queries.
@pytest.mark.parametrize("heads,n_tok", [(32, 768 + r) for r in (1, 16, 17, 128, 129, 255)] + [(32, 1280 + r) for r in (0, 1, 129, 160)]
                         + [(32, 2304 + r) for r in (1, 129)] + [(4, r) for r in (6, 64, 65, 129, 300)])
@pytest.mark.parametrize("sigma,lse", [(1, False), (2, True)])
def test_rows_of_the_last_item(heads, n_tok, sigma, lse):
    wl = inputs.Workload("items", 1, 1, n_tok - 5, 5, heads, 64, sigma, 1, 2, "iid")
    params, ocfg, layer, Q, K, V, O = _run_gpu(wl, seed=3, want_lse=lse)
    _check_attn(ocfg, Q, _host(K), _host(V), O, lse=layer.lse)


# keys 111, 112, 113, 224 and, past the 64 steps after which the row sums move on, 64 x 112 - 1, 64 x 112, 65 x 112 + 1
@pytest.mark.parametrize("n_keys", (111, 112, 113, 224, 7167, 7168, 7281))
def test_key_counts_around_a_step(n_keys):
    wl = inputs.Workload("keys", 1, 1, n_keys, 0, 1, 64, 1, 0, 0, "iid")
    _, ocfg, layer, Q, K, V, O = _run_gpu(wl, seed=4, want_lse=True)
    rows = inputs.sample_rows(wl, 300).numpy()
    _check_attn(ocfg, Q, _host(K), _host(V), O, rows=rows, lse=layer.lse)


@pytest.mark.parametrize("sigma,mean_fill", [(4, 2), (4, 0), (1, 2)])   # (1, 2): nothing dropped, the mean pair is zero-filled
def test_layer_call_gives_the_bits_of_its_two_calls(sigma, mean_fill):
    wl = inputs.Workload("layer", 3, 9, 11, 5, 6, 64, sigma, 1, mean_fill, "proj")
    params, _, layer, Q, K, V, O = _run_gpu(wl, seed=5)
    two = P.SubsampledGlobalAttention(params)
    for t in (two.kmean, two.vmean):
        t.fill_(float("nan"))
    two.build_kv(K, V)
    assert torch.equal(two.attend(Q, K, V), O)
    for a, b in ((two.Kc, layer.Kc), (two.Vc, layer.Vc), (two.idx, layer.idx)):
        assert torch.equal(a, b)
    if mean_fill:
        assert torch.equal(two.kmean, layer.kmean) and torch.equal(two.vmean, layer.vmean)
    with pytest.raises(B.AvggtError):   # everything is rejected before anything is enqueued
        B.avggt_layer(params, Q, K, V, layer.Kc, layer.Vc, layer.idx, layer.kmean, layer.vmean, O, None, layer.build_ws, 0,
                      layer.attn_ws, layer.attn_ws.numel(), None)


# 12 frames x 16 heads, tokens per frame with one tile of rows only, with a full item and a last one of 1, 127, 128, 129 or 255
# rows, and with key tails of 1, 16, 17 and 111 of a 112-key step: several items per thread block, tile 1 sitting some out
@pytest.mark.parametrize("L", (100, 113, 257, 383, 384, 385, 511, 240, 223))
def test_frame_items_with_a_short_last_one(L):
    wl = inputs.Workload("frame_items", 12, 1, L - 5, 5, 16, 64, 4, 1, 2, "iid")
    for lse in (False, True):
        run = frame_attn._run(wl, seed=L, want_lse=lse)
        frame_attn._check(*run)


# 54 items per thread block, all of one tile, so that tile 1 never takes part; 6 or 7 in a row behind as many full ones
@pytest.mark.parametrize("L,n_frames", ((100, 500), (261, 62)))
def test_items_that_a_tile_sits_out_in_a_row(L, n_frames):
    wl = inputs.Workload("sit_out", n_frames, 1, L - 5, 5, 16, 64, 4, 1, 2, "iid")
    for lse in (False, True):
        run = frame_attn._run(wl, seed=L, want_lse=lse)
        frame_attn._check(*run, rows=np.arange(0, wl.n_tokens, 23))


# more bytes than L2 holds, so that the short last items follow the full ones of every two frames (of 16 heads) or of each
# (of 32): 13 frames, the last of them on its own, and 6
@pytest.mark.parametrize("n_frames,heads", ((13, 16), (6, 32)))
def test_frame_items_in_windows(n_frames, heads):
    wl = inputs.Workload("frame_windows", n_frames, 37, 37, 5, heads, 64, 4, 1, 2, "iid")
    frame_attn._check(*frame_attn._run(wl, seed=heads))


def test_layer_items_of_two_steps():
    """121 keys, 288 items of 128 rows."""
    wl = inputs.Workload("two_steps", 1, 33, 33, 0, 32, 64, 9, 1, 2, "iid")
    for seed in range(3):
        _, ocfg, _, Q, K, V, O = _run_gpu(wl, seed=seed)
        _check_attn(ocfg, Q, _host(K), _host(V), O)


# 32 heads x 2,400 queries: 320 items of 256 rows, three rounds of the chip, the last of a head with 96 rows; 113 to 224 keys.  A warp
# without rows must not run an item ahead of the others.
@pytest.mark.parametrize("n_keys", (113, 121, 224))
def test_items_of_two_steps_in_three_rounds(n_keys):
    wl = inputs.Workload("two_steps_256", 1, 40, 60, 0, 32, 64, 4, 1, 2, "iid")
    for seed in range(3):
        idx = np.sort(np.random.default_rng(seed).permutation(wl.n_tokens)[:n_keys]).astype(np.int32)
        indexed._check(wl, idx, seed)


# 8,244 and 8,784 keys, 74 and 79 steps: past the step after which the row sums move on; several items per thread block, which the
# groups of the host-buffer path and the shards number differently (an item is the first of its block in one and not in the other)
@pytest.mark.parametrize("n_frames,sigma,diag,mean_fill", [(6, 1, 0, 0), (24, 4, 1, 2)])
def test_bits_do_not_depend_on_the_place_of_an_item(n_frames, sigma, diag, mean_fill):
    wl = inputs.Workload("places", n_frames, 37, 37, 5, 16, 64, sigma, diag, mean_fill, "proj")
    params, _, layer, Q, K, V, O = _run_gpu(wl, seed=2)
    hQ, hK, hV = (t.cpu().pin_memory() for t in (Q, K, V))
    hO = torch.empty_like(hQ).pin_memory()
    for n_chunks in (1, 3, 6):
        hO.fill_(float("nan"))
        layer.forward_host(hQ, hK, hV, hO, n_chunks=n_chunks)
        layer.check_status()
        assert torch.equal(hO, O.cpu()), n_chunks
    L = wl.tokens_per_frame
    for world in (2, 5):
        for f0, f1 in (sharded.shard_frames(n_frames, world, r) for r in range(world)):
            part = P.make_params(f1 - f0, 37, 37, 5, 16, 64, sigma, diag=diag, mean_fill=mean_fill)
            sl = slice(f0 * L, f1 * L)
            out = torch.full_like(Q[sl], float("nan"))
            P.avggt_global_attn_shard(part, layer.M, layer.n_dropped, Q[sl], K[sl], V[sl], layer.Kc, layer.Vc, layer.kmean,
                                      layer.vmean, out, None, layer.attn_ws, layer.attn_ws.numel())
            layer.check_status()
            assert torch.equal(out, O[sl]), (world, f0)
