"""The time-out path of the attention kernel, exercised without hanging or faulting anything.

Every device-side wait of the kernel is bounded: when one runs out, the thread block records
(code, block, site, iteration) in the workspace's status block, raises a block-wide abort flag,
lets its roles leave in order (copies in flight land, issued tensor-core work completes, tensor
memory is freed) and the other blocks begin no further work item; `avggt_check_status` then returns
AVGGT_ERR_DEVICE_TIMEOUT.  A second build of the same sources (`libavggt_waittest.so`: a 0.5 ms
limit, and the first thread block's producer leaves out one K tile, i.e. a flag that nothing
sets) makes such a wait run out.  The product library does not contain that switch.
"""

import ctypes

import numpy as np
import pytest
import torch

import paper_2512_02541_b200 as P
from oracle import avggt_oracle as orc
from paper_2512_02541_b200 import binding, build, inputs

pytestmark = pytest.mark.gpu


def _forward(L, params, Q, K, V, layer, O):
    """build_kv + global_attn through the library handle L, on the layer's buffers."""
    vp = ctypes.c_void_p
    st = vp(torch.cuda.current_stream().cuda_stream)
    p = ctypes.byref(params)
    rc = L.avggt_build_kv(p, vp(K.data_ptr()), vp(V.data_ptr()), vp(layer.Kc.data_ptr()), vp(layer.Vc.data_ptr()),
                          vp(layer.idx.data_ptr()), vp(layer.kmean.data_ptr()), vp(layer.vmean.data_ptr()),
                          vp(layer.build_ws.data_ptr()), layer.build_ws.numel(), st)
    assert rc == 0
    rc = L.avggt_global_attn(p, vp(Q.data_ptr()), vp(K.data_ptr()), vp(V.data_ptr()), vp(layer.Kc.data_ptr()),
                             vp(layer.Vc.data_ptr()), vp(layer.kmean.data_ptr()), vp(layer.vmean.data_ptr()),
                             vp(O.data_ptr()), None, vp(layer.attn_ws.data_ptr()), layer.attn_ws.numel(), st)
    assert rc == 0
    torch.cuda.synchronize()
    detail = (ctypes.c_uint32 * 4)()
    return L.avggt_check_status(vp(layer.attn_ws.data_ptr()), detail), tuple(detail)


def test_a_wait_that_runs_out_is_reported_and_the_context_stays_usable():
    # 100 frames of 261 tokens, 16 heads: 1632 work items of 119 key steps each, eleven or twelve of about 0.12 ms for each of
    # 148 thread blocks, so that the first block's wait (0.5 ms) runs out while the others have most of theirs before them
    wl = inputs.Workload("wait_limit", 100, 16, 16, 5, 16, 64, 2, 1, 2, "iid")
    params = P.make_params(wl.n_frames, wl.grid_h, wl.grid_w, wl.n_special, wl.n_heads, wl.head_dim, wl.sigma,
                           diag=wl.diag, mean_fill=wl.mean_fill)
    Q, K, V = inputs.make_qkv(wl, seed=0, device="cuda")
    layer = P.SubsampledGlobalAttention(params)
    O = torch.full_like(Q, float("nan"))

    broken = binding.load_library(build.build_wait_test())
    code, detail = _forward(broken, params, Q, K, V, layer, O)
    assert code == binding.AVGGT_ERR_DEVICE_TIMEOUT
    flag, block, site, iteration = detail
    assert flag == 1 and block == 0                       # the first thread block gave up ...
    # ... in whichever of its roles had waited longest on the consequences of the missing K tile: the producer
    # on a ring stage that is never released (sites 10, 11), an MMA issuer on the tile itself (24, 25) or a
    # softmax warp on the scores of step 1 (40, 41); all within the item's first six steps
    assert site in (10, 11, 24, 25, 40, 41) and iteration <= 5
    # the items of the last head were not begun: the blocks had seen the time-out by then
    assert torch.isnan(O[:, wl.n_heads - 1].float()).any()

    # the same workspace and buffers through the product library right afterwards: correct output
    good = binding.lib()
    O.fill_(float("nan"))
    code, detail = _forward(good, params, Q, K, V, layer, O)
    assert code == 0 and detail[0] == 0
    assert torch.isfinite(O.float()).all()
    ocfg = orc.SGAConfig(wl.n_frames, wl.grid_h, wl.grid_w, wl.n_special, wl.n_heads, wl.head_dim, wl.sigma,
                         diag=bool(wl.diag), mean_fill=wl.mean_fill)
    Qh, Kh, Vh = (t.float().cpu().numpy() for t in (Q, K, V))
    rows = inputs.sample_rows(wl, 256).numpy()
    want = orc.global_attn_blocked(ocfg, Qh, Kh, Vh, rows)
    err = np.abs(O[torch.as_tensor(rows, device="cuda")].float().cpu().numpy().astype(np.float64) - want)
    assert err.max() <= 2e-2 and err.mean() <= 2e-3


def _small(mean_fill):
    # 13,740 tokens of 16 heads, a quarter retained: 1,718 tiles of 8 tokens, or 458 of 8 compact rows, over 296 thread blocks
    wl = inputs.Workload("wait_limit_small", 10, 37, 37, 5, 16, 64, 4, 1, mean_fill, "iid")
    params = P.make_params(wl.n_frames, wl.grid_h, wl.grid_w, wl.n_special, wl.n_heads, wl.head_dim, wl.sigma,
                           diag=wl.diag, mean_fill=wl.mean_fill)
    return params, P.SubsampledGlobalAttention(params), inputs.make_qkv(wl, seed=1, device="cuda")


@pytest.mark.parametrize("mean_fill", (2, 0))   # tiles of tokens, tiles of compact rows
def test_a_compaction_that_lost_a_tile_shows(mean_fill):
    params, layer, (Q, K, V) = _small(mean_fill)
    vp = ctypes.c_void_p
    st = vp(torch.cuda.current_stream().cuda_stream)
    broken = binding.load_library(build.build_wait_test())
    buffers = (layer.Kc, layer.Vc, layer.idx, layer.kmean, layer.vmean)
    for t in buffers[:2]:
        t.zero_()
    args = [vp(t.data_ptr()) for t in (K, V) + buffers]
    assert broken.avggt_build_kv(ctypes.byref(params), *args, vp(layer.build_ws.data_ptr()), layer.build_ws.numel(), st) == 0
    torch.cuda.synchronize()
    got = [t.clone() for t in buffers]

    layer.build_kv(K, V)   # the product library, the same buffers
    layer.check_status()
    lost = torch.isnan(got[0].float()).any(dim=2).any(dim=0)
    assert 0 < int(lost.sum()) < layer.M // 4   # what the first thread block had before it
    for bad, good in zip(got[:2], buffers[:2]):
        assert torch.isfinite(good.float()).all()
        assert torch.isnan(bad[:, lost].float()).all() and torch.equal(bad[:, ~lost], good[:, ~lost])
    if mean_fill:
        assert torch.isnan(got[3]).all() and torch.isnan(got[4]).all() and torch.isfinite(layer.kmean).all()


@pytest.mark.parametrize("mean_fill", (2, 0))
def test_the_layer_reports_a_compaction_that_lost_a_tile(mean_fill):
    params, layer, (Q, K, V) = _small(mean_fill)
    vp = ctypes.c_void_p
    st = vp(torch.cuda.current_stream().cuda_stream)
    broken = binding.load_library(build.build_wait_test())
    O = torch.empty_like(Q)
    args = [vp(t.data_ptr()) for t in (Q, K, V, layer.Kc, layer.Vc, layer.idx, layer.kmean, layer.vmean, O)]
    assert broken.avggt_layer(ctypes.byref(params), *args, None, vp(layer.build_ws.data_ptr()), layer.build_ws.numel(),
                              vp(layer.attn_ws.data_ptr()), layer.attn_ws.numel(), st) == 0
    torch.cuda.synchronize()
    detail = (ctypes.c_uint32 * 4)()
    assert broken.avggt_check_status(vp(layer.attn_ws.data_ptr()), detail) == binding.AVGGT_ERR_DEVICE_TIMEOUT
    assert tuple(detail)[:3] == (1, 0, 90)
    layer.forward(Q, K, V)
    layer.check_status()
