"""GPU: the CUDA-core layer kernels (fp32 verification mode, and a bf16 expert whose dims the
tensor-core kernels do not tile) against the fp64 oracle, at the edges of their tiles: one to
many 16-token row tiles, K below and above the 128-wide steps and not a multiple of 4, an odd MLP
width, head dims of one to eight 32-lane groups, one and four heads per attention block, and the
embedding's blocks of several tokens."""

import numpy as np
import pytest
import torch

import oracle
from gpu_util import BF16_REL_L2, make_expert, oracle_denoise, gpu_denoise
from synth import TINY, make_requests, make_weights

pytestmark = pytest.mark.gpu

# (overrides, batch, prefix, chunk, steps)
CASES = [
    (dict(), 1, 1, 1, 1),
    (dict(), 3, 64, 14, 2),
    (dict(width=32, n_heads=1, head_dim=32, mlp_dim=33), 2, 5, 16, 2),      # odd K: scalar loads
    (dict(width=160, n_heads=3, head_dim=96, mlp_dim=130), 1, 37, 9, 1),    # K % 4 != 0 in down only
    (dict(width=512, n_heads=8, head_dim=256, mlp_dim=96), 2, 130, 33, 1),  # four heads per block
    (dict(width=64, n_heads=4, head_dim=32, mlp_dim=64, action_dim=40, state_dim=33), 50, 3, 50, 1),
    (dict(rope_base=0.0), 1, 33, 8, 2),
    (dict(), 20, 7, 50, 1),                                                 # 64 x 64 tiles for gate/up
    (dict(), 31, 7, 50, 1),                                                 # and for QKV and O
]


@pytest.mark.parametrize("over,B,P,C,N", CASES)
def test_fp32_matches_oracle(over, B, P, C, N):
    cfg = TINY.with_(**over)
    w = make_weights(cfg, 3, mod_bias_std=0.3)
    r = make_requests(cfg, 5, B, P, C)
    ex = make_expert(cfg, w, max_batch=B, max_prefix=P, max_chunk=C, max_steps=N)
    got = gpu_denoise(ex, cfg, r, N)
    ex.close()
    pick = range(B) if B < 8 else (0, B - 1)
    ref = oracle_denoise(cfg, w, r, N, pick)
    # fp32 products of up to ~1000 terms summed in another order: about 1e-6 of the values (O(1)).
    assert np.abs(got[list(pick)] - ref).max() <= 2e-5


def test_bf16_outside_the_tensor_core_tiling():
    cfg = TINY.with_(precision="bf16", width=96, n_heads=2, head_dim=64, mlp_dim=90)
    w = make_weights(cfg, 3, mod_bias_std=0.3)
    r = make_requests(cfg, 5, 2, 70, 20)
    ex = make_expert(cfg, w, max_batch=2, max_prefix=70, max_chunk=20, max_steps=2)
    got = gpu_denoise(ex, cfg, r, 2)
    ex.close()
    ref = oracle_denoise(cfg, w, r, 2)
    assert np.linalg.norm(got - ref) <= BF16_REL_L2 * np.linalg.norm(ref)


def test_correction_items_fp32():
    cfg = TINY
    w = make_weights(cfg, 3, mod_bias_std=0.3)
    r = make_requests(cfg, 5, 2, 65, 20)
    from synth import make_correction
    items = make_correction(cfg, 5, 2, 3, std=0.5)
    ex = make_expert(cfg, w, max_batch=2, max_prefix=65, max_chunk=20, max_steps=2)
    ex.set_correction(torch.from_numpy(items).cuda())
    got = gpu_denoise(ex, cfg, r, 2)
    ex.close()
    ref = oracle.denoise_batch(r["noise"], r["state"], 2, r["prefix_k"], r["prefix_v"], w, cfg, corr=items)
    assert np.abs(got - ref).max() <= 2e-5


# The final norm and output product at every number of rows a block takes (one with one or two blocks on an
# SM, four, eight), at widths of less than and more than the steps fetched ahead: a request's bits do not
# depend on it.
@pytest.mark.parametrize("W", [256, 1120])
def test_final_rows_same_bits_in_every_block_shape(monkeypatch, W):
    monkeypatch.setenv("JPI_BATCH_INVARIANT", "1")
    cfg = TINY.with_(n_layers=1, width=W, n_heads=1, head_dim=32, mlp_dim=64)
    w, P, C = make_weights(cfg, 3, mod_bias_std=0.3), 3, 50
    ex = make_expert(cfg, w, max_batch=26, max_prefix=P, max_chunk=C, max_steps=1)
    got = {B: gpu_denoise(ex, cfg, make_requests(cfg, 5, B, P, C), 1) for B in (1, 3, 4, 6, 7, 26)}
    ex.close()
    for B in (3, 4, 6, 7):
        assert np.array_equal(got[B], got[26][:B]), B
    assert np.array_equal(got[1], got[26][:1])
    ref = oracle_denoise(cfg, w, make_requests(cfg, 5, 26, P, C), 1, (0, 25))
    assert np.abs(got[26][[0, 25]] - ref).max() <= 2e-5
