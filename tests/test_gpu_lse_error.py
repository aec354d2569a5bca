"""How far the log-sum-exp is from 64 bits, by the key that the softmax is concentrated on."""

import numpy as np
import pytest
import torch

import paper_2512_02541_b200 as P

pytestmark = pytest.mark.gpu


def test_columns_whose_exponentials_are_polynomials():
    """Frames of 112 tokens, one full key step; token j is 16 times a unit vector (or its negative), so that its own key takes all of
    its softmax (raw scores 256, 0 and -256; the others weigh 1e-12 together) and the log-sum-exp is 256 / 8.  A key in a block of
    eight columns from the special-function unit leaves the roundings of the score, the scale, the product and the result:
    2^-24 of 32 each, 7.6e-6 together.  One in a block from the polynomial adds up to 7.5e-5; there are two such blocks in fourteen."""
    L, frames, heads = 112, 3, 2
    params = P.make_params(frames, 1, L, 0, heads, 64, 4)
    token = torch.zeros((L, 64))
    j = torch.arange(L)
    token[j, j % 64] = torch.where(j < 64, 16.0, -16.0)
    X = token.repeat(frames, 1).reshape(frames * L, 1, 64).expand(-1, heads, -1).to(device="cuda", dtype=torch.bfloat16).contiguous()
    layer = P.SubsampledGlobalAttention(params, want_lse=True)
    layer.frame_attend(X, X, X)
    layer.check_status()
    scores = token.double() @ token.double().T / 8
    want = torch.logsumexp(scores, dim=1).numpy()
    err = np.abs(layer.lse.cpu().numpy().astype(np.float64).reshape(frames, L, heads) - want[None, :, None])
    by_block = err.max(axis=(0, 2)).reshape(L // 8, 8).max(axis=1)
    assert by_block.max() <= 7.5e-5 + 1e-5
    assert (by_block > 1e-5).sum() <= 2, by_block
