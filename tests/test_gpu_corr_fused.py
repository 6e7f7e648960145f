"""GPU: the correction module's launches that take their neighbours in (LayerNorm, four-token attention,
position table, join, query segment and confidence inside the streamed products) against the fp64
oracle, on both sides of every rule that chooses them: rows per call (batch and Delta), item counts
other than four, a head dim that is no power of two, VLM tokens around the 32-token chunks, and more
than 32 query rows (heads x items). A request's bits must not depend on its batch."""

import numpy as np
import pytest

import oracle.correction as oc
from synth import PI05_CORRECTION
from tests.test_gpu_corr import _close, _setup

pytestmark = pytest.mark.gpu

BASE = PI05_CORRECTION.with_(width=256, n_heads=2, head_dim=128, mlp_dim=512, d_vlm=320, max_delta=24)
CONFIGS = {
    "four": BASE,
    "three_items": BASE.with_(n_items=3),
    "head96": BASE.with_(width=192, n_heads=2, head_dim=96),
    "many_rows": BASE.with_(n_heads=8, head_dim=32, n_items=5),
    "head32": BASE.with_(n_heads=8, head_dim=32),
}


@pytest.mark.parametrize("name", CONFIGS)
@pytest.mark.parametrize("B,T,delta", [(1, 31, 1), (2, 33, 8), (3, 64, 5), (5, 65, 4), (4, 1, 17)])
def test_fused_launches(name, B, T, delta):
    import torch
    cfg = CONFIGS[name]
    mod, w, inp, dev = _setup(cfg, 301, B, T, delta, max_batch=8, max_tokens=80)
    z = mod.compress(dev["h_vlm"])
    h, c = mod.predict(z, dev["actions"])
    b = B - 1
    z1 = mod.compress(dev["h_vlm"][b:])
    h1, c1 = mod.predict(z1, dev["actions"][b:])
    torch.cuda.synchronize()
    assert torch.equal(z[b:], z1) and torch.equal(h[b:], h1) and torch.equal(c[b:], c1)
    want_z = oc.compress_batch(inp["h_vlm"], w, cfg)
    _close(z.cpu().numpy(), want_z, f"fused {name}: state")
    want_h, want_c = oc.correction_batch(want_z, inp["actions"], w, cfg)
    _close(h.cpu().numpy(), want_h, f"fused {name}: predicted")
    assert np.abs(c.cpu().numpy() - want_c).max() <= 5e-4
    mod.close()
