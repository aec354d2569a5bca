"""The two compaction kernels (few tokens: a cluster of thread blocks per head; many: a warp per row) over the head counts that
select their variants, against the oracle: bit copies, indices, and the mean pair."""

import pytest
import torch

import paper_2512_02541_b200 as P
from paper_2512_02541_b200 import inputs

from test_gpu_parity import _cfgs, _check_build

pytestmark = pytest.mark.gpu


# 1 to 8 chunks of 16 bytes per lane and row in the many-token kernel; clusters of 8, 4, 2 blocks in the other, whose
# limit lies at 11,520 tokens for up to 6 heads, 5,760 up to 18, 2,880 above; 12,300 and 1,230 tokens, not a multiple of any group
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
