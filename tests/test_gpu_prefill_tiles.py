"""GPU: the prefill's fused QKV epilogue, its stream-K residual products and its attention key splits at
the edges of their tiles, against the fp64 oracle: rows around one and two 128-row tiles, two requests
whose rows share a tile, both fused head dims (one and two head sections per 256-column tile, an odd
number of sections at 128), k-block counts that cut CTAs across tiles, and a request stride wider than
the prefix."""

import numpy as np
import pytest

import oracle.prefill as pf
from synth import GEMMA2B, make_llm_weights, make_prefix_embeddings

pytestmark = pytest.mark.gpu

# bf16 operands: the tolerance of tests/test_gpu_prefill.py.
REL_L2 = 2e-2
WIDE = GEMMA2B.with_(n_layers=2, width=512, n_heads=4, head_dim=256, mlp_dim=4096 + 72)   # down: 66 k-blocks
ODD = GEMMA2B.with_(n_layers=2, width=320, n_heads=3, head_dim=128, mlp_dim=1000)         # 5 sections of 128


@pytest.mark.parametrize("cfg", [WIDE, ODD], ids=["wide", "odd"])
@pytest.mark.parametrize("B,P,pad", [(1, 1, 0), (1, 127, 3), (2, 64, 0), (1, 129, 0), (2, 100, 8), (1, 300, 0)])
def test_prefill_tiles(cfg, B, P, pad):
    import torch
    from tests.gpu_util import errors, lib
    lib()
    from paper_2607_12659_gb300 import prefill
    w = make_llm_weights(cfg, 131, std=0.05, norm_std=0.1)
    x = make_prefix_embeddings(cfg, 132 + P, B, P)
    pre = prefill.Prefill(cfg, w, max_batch=B, max_prefix=P)
    L, D = cfg.n_layers, cfg.head_dim
    K = torch.full((L, B, P + pad, D), 7.0, dtype=torch.bfloat16, device="cuda")
    V = torch.full_like(K, 7.0)
    out = pre.run(torch.from_numpy(x).cuda(), [K[l].data_ptr() for l in range(L)],
                  [V[l].data_ptr() for l in range(L)], (P + pad) * D)
    torch.cuda.synchronize()
    pre.device_status()
    Kw, Vw, want = pf.prefill_batch(x, w, cfg)
    for l in range(L):
        for got, ref, what in ((K, Kw, "K"), (V, Vw, "V")):
            _, rel = errors(got[l, :, :P].float().cpu().numpy(), ref[l])
            assert rel <= REL_L2, f"{what} layer {l}: rel-L2 {rel:.3g}"
            assert bool((got[l, :, P:] == 7.0).all()), f"{what} layer {l}: rows past the prefix were written"
    _, rel = errors(out.cpu().numpy(), want)
    assert rel <= REL_L2, f"final output rel-L2 {rel:.3g}"
    assert np.isfinite(out.cpu().numpy()).all()
    pre.close()
