"""GPU: the prefix copy into the KV store, bit for bit, at the edges of its chunks: source types,
store types, sources that are not 16-byte aligned, ragged prefix lengths, several requests, and more
layers than one launch carries."""

import numpy as np
import pytest
import torch

from paper_2607_12659_gb300 import jpi
from synth import TINY, make_weights

pytestmark = pytest.mark.gpu


class _View:
    def __init__(self, ptr, shape, strides, typestr):
        self.__cuda_array_interface__ = {"shape": shape, "strides": strides, "typestr": typestr, "version": 3,
                                         "data": (ptr, False)}


def _store(ex, layer, B, P, D, bf16):
    k, v, stride = jpi.jpi_prefix_kv_ptr(ex.handle, layer)
    size = 2 if bf16 else 4
    out = []
    for p in (k, v):
        t = torch.as_tensor(_View(p, (B, P, D), (stride * size, D * size, size), "<i2" if bf16 else "<f4"),
                            device="cuda")
        out.append((t.view(torch.bfloat16) if bf16 else t).clone())
    return out


@pytest.mark.parametrize("precision,src", [("bf16", torch.bfloat16), ("bf16", torch.float32),
                                           ("fp32", torch.float32), ("fp32", torch.bfloat16)])
@pytest.mark.parametrize("layers,B,P,shift", [(2, 1, 1, 0), (2, 3, 129, 0), (2, 2, 33, 1), (1, 5, 1030, 0),
                                              (66, 1, 3, 0)])
def test_prefix_store_holds_the_source(precision, src, layers, B, P, shift):
    cfg = TINY.with_(n_layers=layers, width=32, n_heads=1, head_dim=32, mlp_dim=32, time_dim=4, precision=precision)
    ex = jpi.Expert(cfg, make_weights(cfg, 0), max_batch=B, max_prefix=P + 5, max_chunk=2, max_steps=1)
    D = cfg.head_dim
    g = torch.Generator(device="cuda").manual_seed(1)
    n = B * P * D
    ks, vs = ([torch.randn(n + shift, generator=g, device="cuda").to(src)[shift:] for _ in range(layers)]
              for _ in range(2))
    jpi.jpi_set_prefix_kv(ex.handle, ks, vs, B, P, src == torch.float32)
    torch.cuda.synchronize()
    bf16 = precision == "bf16"
    want_type = torch.bfloat16 if bf16 else torch.float32
    for l in range(layers):
        for got, want in zip(_store(ex, l, B, P, D, bf16), (ks[l], vs[l])):
            assert torch.equal(got, want.view(B, P, D).to(want_type)), (l, np.array(got.shape))
    ex.close()
