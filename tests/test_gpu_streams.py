"""GPU: the wrappers' calls on a stream other than the current one. The inputs need a conversion, whose
temporaries nobody holds once the call has returned; the call is still waiting behind other work on its
stream when the current stream allocates and overwrites memory of every size it used. The results are those of the
same call on the current stream, bit for bit."""

import numpy as np
import pytest
import torch

from synth import GEMMA2B, PI05_CORRECTION, TINY, make_llm_weights, make_requests, make_weights
from tests.gpu_util import make_expert
from tests.test_gpu_corr import _setup

pytestmark = pytest.mark.gpu


def _strided(t):
    """The values of t in a tensor that is not contiguous."""
    return t.transpose(0, -1).contiguous().transpose(0, -1) if t.dim() > 1 and t.shape[0] > 1 and t.shape[-1] > 1 \
        else torch.stack((t, t), -1)[..., 0]


def _on_a_busy_stream(call, sizes, raw):
    """call(stream) on a stream that is busy for some milliseconds; meanwhile the current stream writes
    over fresh tensors of the given sizes (bytes), again and again."""
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        torch.cuda._sleep(20_000_000)
    out = call(side.cuda_stream if raw else side)
    junk = [torch.full((n,), 255, dtype=torch.uint8, device="cuda") for n in sizes for _ in range(4)]
    torch.cuda.synchronize()
    del junk
    return out


@pytest.mark.parametrize("raw", [False, True])
def test_corrector(raw):
    cfg = PI05_CORRECTION.with_(width=256, n_heads=2, head_dim=128, mlp_dim=512, d_vlm=320, max_delta=24)
    mod, w, inp, dev = _setup(cfg, 401, 3, 64, 8, max_batch=4, max_tokens=80)
    vlm, act = _strided(dev["h_vlm"]), _strided(dev["actions"])
    assert not vlm.is_contiguous() and not act.is_contiguous()
    z = mod.compress(vlm)
    zs = _strided(z)
    h, c = mod.predict(zs, act)
    torch.cuda.synchronize()

    def call(stream):
        z2 = mod.compress(vlm, stream=stream)
        return (z2, *mod.predict(zs, act, stream=stream))
    sizes = [t.numel() * t.element_size() for t in (vlm, zs, act, z, h, c)]
    for _ in range(3):
        for got, want in zip(_on_a_busy_stream(call, sizes, raw), (z, h, c)):
            assert torch.equal(got, want)
    mod.close()


@pytest.mark.parametrize("raw", [False, True])
def test_expert(raw):
    cfg, B, P, C, N = TINY, 2, 40, 6, 2
    ex = make_expert(cfg, make_weights(cfg, 402), max_batch=B, max_prefix=P, max_chunk=C, max_steps=N)
    r = make_requests(cfg, 403, B, P, C)
    k, v = (_strided(torch.from_numpy(r[n]).cuda()) for n in ("prefix_k", "prefix_v"))
    items = _strided(torch.randn(B, 3, cfg.width, device="cuda", generator=torch.Generator("cuda").manual_seed(4)))
    state, noise = torch.from_numpy(r["state"]).cuda(), torch.from_numpy(r["noise"]).cuda()

    def call(stream):
        ex.set_prefix_kv(k, v, stream=stream)
        ex.set_correction(items, stream=stream)
        return (ex.denoise(state, noise, N, stream=stream), *ex.forward(state, noise, 0.3, stream=stream))
    want = call(None)
    torch.cuda.synchronize()
    sizes = [t.numel() * t.element_size() for t in (k, items, *want)]
    for _ in range(3):
        for got, ref in zip(_on_a_busy_stream(call, sizes, raw), want):
            assert torch.equal(got, ref)
    ex.close()


@pytest.mark.parametrize("raw", [False, True])
def test_prefill(raw):
    from paper_2607_12659_gb300 import prefill
    cfg, B, P = GEMMA2B.with_(n_layers=2, width=320, n_heads=3, head_dim=128, mlp_dim=1000), 2, 50
    pre = prefill.Prefill(cfg, make_llm_weights(cfg, 404, std=0.05), max_batch=B, max_prefix=P)
    x = _strided(torch.randn(B, P, cfg.width, device="cuda", generator=torch.Generator("cuda").manual_seed(5)))
    want = pre.into_tensors(x)
    torch.cuda.synchronize()
    sizes = [t.numel() * t.element_size() for t in (x, *want)]
    for _ in range(3):
        for got, ref in zip(_on_a_busy_stream(lambda s: pre.into_tensors(x, stream=s), sizes, raw), want):
            assert torch.equal(got, ref)
    pre.close()
    assert np.isfinite(want[2].cpu().numpy()).all()
