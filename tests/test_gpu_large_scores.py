"""Scores far beyond what a model produces: the softmax is then one key's value, and stays finite as long as a score's own
rounding (2^-24 of it, in log2 units) is small against the range of an exponential."""

import numpy as np
import pytest
import torch

import paper_2512_02541_b200 as P
from oracle import avggt_oracle as orc
from paper_2512_02541_b200 import inputs

from test_gpu_parity import _cfgs, _check_attn, _host

pytestmark = pytest.mark.gpu


# Q and K scaled by sqrt(magnitude): scores with a standard deviation of 4e4 log2 units at 1e4 to 4e8 at 1e8, so that the references lie
# on either side of the size (2^20) from which a row looks at every step; one ordinary row in sixteen among them.  (Sizes at
# which no row's two largest scores lie within their rounding of each other.)
@pytest.mark.parametrize("magnitude", (1e4, 1e5, 3e6, 1e7, 1e8))
@pytest.mark.parametrize("sigma,diag,mean_fill", [(4, 1, 2), (1, 0, 0)])
@pytest.mark.parametrize("want_lse", (False, True))
def test_large_scores(magnitude, sigma, diag, mean_fill, want_lse):
    wl = inputs.Workload("large", 4, 16, 16, 5, 4, 64, sigma, diag, mean_fill, "iid")
    params, ocfg = _cfgs(wl)
    Q, K, V = inputs.make_qkv(wl, seed=3, device="cuda")
    Q, K = (Q.float() * magnitude ** 0.5).bfloat16(), (K.float() * magnitude ** 0.5).bfloat16()
    Q[::16] = (Q[::16].float() / magnitude).bfloat16()   # ordinary rows share a warp with the others
    layer = P.SubsampledGlobalAttention(params, want_lse=want_lse)
    O = layer.forward(Q, K, V)
    layer.check_status()
    _check_attn(ocfg, Q, _host(K), _host(V), O)
    F = layer.frame_attend(Q, K, V)
    layer.check_status()
    want = orc.frame_attn(ocfg, _host(Q), _host(K), _host(V))
    assert np.abs(F.float().cpu().numpy().astype(np.float64) - want).max() <= 2e-2
