"""GPU: the large-M projection kernel with the tokens on the MMA's rows, forced on every projection,
against the fp64 oracle at the edges of its tiles: token counts around one and two tiles (126 tokens
for the norm-fed kinds, 128 for the residual kinds), an odd number of 128-row weight tiles (the
second half of the last 256-row tile is padding) and both tile widths of the norm-fed kinds."""

import pytest

import oracle
from synth import ExpertConfig, make_requests, make_weights
from tests.gpu_util import assert_close, errors, lib, make_expert, to_dev_kv

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

# Weight tiles per projection (QKV, O, gate/up, down): 4, 1, 1, 1; one head of 128: 3, 2, 8, 2.
ODD = ExpertConfig(n_layers=2, width=128, n_heads=2, head_dim=128, mlp_dim=64, action_dim=7, state_dim=7,
                   time_dim=64, precision="bf16")
ONE_HEAD = ODD.with_(width=256, n_heads=1, mlp_dim=512)


@pytest.mark.parametrize("cfg", [ODD, ONE_HEAD], ids=["odd_tiles", "one_head"])
@pytest.mark.parametrize("tile_n", ["128", "256"])
@pytest.mark.parametrize("B,C", [(1, 1), (2, 62), (1, 126), (3, 41), (1, 127), (1, 128), (3, 84), (4, 63)])
def test_tokens_on_rows_kernel(monkeypatch, cfg, B, C, tile_n):
    lib()
    monkeypatch.setenv("JPI_BIG_GEMM_MIN_TOKENS", "1")
    monkeypatch.setenv("JPI_BIG_RESID_ROWS", "1")
    monkeypatch.setenv("JPI_BIG_TILE_N", tile_n)
    P, t = 70, 0.4
    w = make_weights(cfg, 77, mod_bias_std=0.3)
    r = make_requests(cfg, 78 + B + C, B, P, C)
    ex = make_expert(cfg, w, max_batch=B, max_prefix=P, max_chunk=C, max_steps=1)
    try:
        ex.set_prefix_kv(*to_dev_kv(r, cfg))
        v, h = ex.forward(torch.from_numpy(r["state"]).cuda(), torch.from_numpy(r["noise"]).cuda(), t)
        torch.cuda.synchronize()
        ex.device_status()
    finally:
        ex.close()
    want_v, want_h = oracle.forward_batch(r["noise"], r["state"], t, r["prefix_k"], r["prefix_v"], w, cfg)
    assert_close(v.cpu().numpy(), want_v, cfg, f"rows kernel B{B} C{C}")
    # bf16 operands (2^-9 each) of four projections a layer, two layers.
    _, rel = errors(h.cpu().numpy(), want_h)
    assert rel <= 1e-2, f"hidden rel-L2 {rel:.3g}"
