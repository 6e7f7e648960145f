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


# Query weights larger than the MLP's: host tensors pass through one staging buffer.
@pytest.mark.parametrize("over", [dict(width=64, n_heads=8, head_dim=128, mlp_dim=8),
                                  dict(width=32, n_heads=1, head_dim=64, mlp_dim=16)])
def test_prefill_of_more_head_than_mlp_features(over):
    from tests.gpu_util import errors, lib
    import torch
    lib()
    from paper_2607_12659_gb300 import prefill
    cfg, P = GEMMA2B.with_(n_layers=2, **over), 40
    w = make_llm_weights(cfg, 171, std=0.05, norm_std=0.1)
    x = make_prefix_embeddings(cfg, 172, 1, P)
    pre = prefill.Prefill(cfg, w, max_batch=1, max_prefix=P)
    K, V, out = pre.into_tensors(torch.from_numpy(x).cuda())
    torch.cuda.synchronize()
    pre.device_status()
    pre.close()
    for got, ref in zip((K, V, out), pf.prefill_batch(x, w, cfg)):
        _, rel = errors(got.float().cpu().numpy(), np.stack(ref) if isinstance(ref, list) else ref)
        assert rel <= REL_L2, f"rel-L2 {rel:.3g}"


# Value destinations that are only element-aligned, which the attention's bulk copies cannot read: taken
# where the request stride is no multiple of the head dim (the per-request products), refused otherwise.
@pytest.mark.parametrize("cfg", [WIDE, ODD], ids=["wide", "odd"])
@pytest.mark.parametrize("shift", [0, 1, 2, 8])
def test_prefill_value_destinations_at_any_element(cfg, shift):
    import torch
    from tests.gpu_util import errors, lib
    lib()
    from paper_2607_12659_gb300 import prefill
    B, P, L, D = 2, 100, cfg.n_layers, cfg.head_dim
    stride = P * D + 8
    w = make_llm_weights(cfg, 141, std=0.05, norm_std=0.1)
    x = make_prefix_embeddings(cfg, 142, B, P)
    pre = prefill.Prefill(cfg, w, max_batch=B, max_prefix=P)
    K = torch.full((L, B * stride), 7.0, dtype=torch.bfloat16, device="cuda")
    V = torch.full((L, B * stride + 16), 7.0, dtype=torch.bfloat16, device="cuda")
    out = pre.run(torch.from_numpy(x).cuda(), [K[l].data_ptr() for l in range(L)],
                  [V[l, shift:].data_ptr() for l in range(L)], stride)
    torch.cuda.synchronize()
    pre.device_status()
    Kw, Vw, want = pf.prefill_batch(x, w, cfg)
    for l in range(L):
        for got, ref, what in ((K[l], Kw[l], "K"), (V[l, shift:shift + B * stride], Vw[l], "V")):
            rows = got.view(B, stride).float().cpu().numpy()
            _, rel = errors(rows[:, :P * D].reshape(B, P, D), ref)
            assert rel <= REL_L2, f"{what} layer {l}: rel-L2 {rel:.3g}"
            assert (rows[:, P * D:] == 7.0).all(), f"{what} layer {l}: written past the prefix"
        assert bool((V[l, :shift] == 7.0).all()) and bool((V[l, shift + B * stride:] == 7.0).all())
    _, rel = errors(out.cpu().numpy(), want)
    assert rel <= REL_L2, f"final output rel-L2 {rel:.3g}"
    pre.close()


@pytest.mark.parametrize("which,pad,shift", [("k", 0, 4), ("v", 0, 4), ("k", 8, 4)])
def test_prefill_refuses_a_misaligned_layer_before_it_runs_any(which, pad, shift):
    import torch
    from tests.gpu_util import lib
    lib()
    from paper_2607_12659_gb300 import prefill
    from paper_2607_12659_gb300.jpi import JpiError
    cfg, P = ODD, 20
    L, D = cfg.n_layers, cfg.head_dim
    pre = prefill.Prefill(cfg, make_llm_weights(cfg, 151, std=0.05), max_batch=1, max_prefix=P)
    x = torch.from_numpy(make_prefix_embeddings(cfg, 152, 1, P)).cuda()
    kv = {n: torch.full((L, P * D + 16), 7.0, dtype=torch.bfloat16, device="cuda") for n in "kv"}
    ptr = {n: [kv[n][l].data_ptr() for l in range(L)] for n in "kv"}
    ptr[which][-1] += 2 * shift
    with pytest.raises(JpiError):
        pre.run(x, ptr["k"], ptr["v"], P * D + pad)
    torch.cuda.synchronize()
    assert bool((kv["k"] == 7.0).all()) and bool((kv["v"] == 7.0).all())
    pre.close()


# The final output at an address that takes no 16-byte stores, from the pieces' sum (many k-blocks a tile)
# and after the product that accumulates in place (few): the same bits as at an aligned address.
@pytest.mark.parametrize("cfg,P", [(ODD, 20), (WIDE, 100), (ODD.with_(mlp_dim=384), 20)])
def test_prefill_final_output_at_any_float(cfg, P):
    import torch
    from tests.gpu_util import lib
    lib()
    from paper_2607_12659_gb300 import prefill
    L, D, W = cfg.n_layers, cfg.head_dim, cfg.width
    pre = prefill.Prefill(cfg, make_llm_weights(cfg, 161, std=0.05), max_batch=1, max_prefix=P)
    x = torch.from_numpy(make_prefix_embeddings(cfg, 162, 1, P)).cuda()
    K = torch.zeros((L, P, D), dtype=torch.bfloat16, device="cuda")
    V = torch.zeros_like(K)
    kp, vp = [K[l].data_ptr() for l in range(L)], [V[l].data_ptr() for l in range(L)]
    outs = []
    for shift in (0, 1, 2):
        buf = torch.full((P * W + 4,), 7.0, device="cuda")
        prefill.jpi_prefill_run(pre.handle, x, True, 1, P, kp, vp, P * D, buf[shift:])
        torch.cuda.synchronize()
        assert bool((buf[:shift] == 7.0).all()) and bool((buf[shift + P * W:] == 7.0).all())
        outs.append(buf[shift:shift + P * W].clone())
    pre.device_status()
    assert torch.equal(outs[0], outs[1]) and torch.equal(outs[0], outs[2])
    assert bool((outs[0] != 7.0).all())
    pre.close()
