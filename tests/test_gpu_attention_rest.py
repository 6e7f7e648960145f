"""GPU: batches one or a few requests past a whole wave of the tcgen05 attention, whose last requests run
in a launch of their own split over the keys, against the fp64 oracle for requests on both sides of
the cut: one (D = 128) and four (D = 256) row blocks per request, the cut's first and last request, and a
rest too large to split (one launch)."""

import pytest

import oracle
from synth import ExpertConfig, make_requests, make_weights
from tests.gpu_util import assert_close, lib, make_expert, to_dev_kv

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

# 8 heads x 51 rows: four row blocks; 2 heads x 6 rows: one.
FOUR = (ExpertConfig(n_layers=1, width=128, n_heads=8, head_dim=256, mlp_dim=128, action_dim=7, state_dim=7,
                     time_dim=64, precision="bf16"), 50, 4)
ONE = (ExpertConfig(n_layers=1, width=128, n_heads=2, head_dim=128, mlp_dim=128, action_dim=7, state_dim=7,
                    time_dim=64, precision="bf16"), 5, 1)


# Below 8 key blocks (P < 398 and 443) and at a rest of 30 there is one launch; from there on four splits, two at
# a rest of 12 from 16 blocks; 40 is a rest of 2 past two whole waves, 78 past three (one launch).
@pytest.mark.parametrize("shape,rest,P", [(FOUR, 1, 300), (FOUR, 9, 230), (FOUR, 12, 1000), (FOUR, 30, 300),
                                          (ONE, 1, 300), (ONE, 37, 250), (FOUR, 1, 397), (FOUR, 1, 398),
                                          (FOUR, 9, 500), (FOUR, 12, 909), (FOUR, 40, 520), (FOUR, 78, 450),
                                          (ONE, 1, 510), (ONE, 37, 630)])
def test_last_requests_split_over_the_keys(shape, rest, P):
    lib()
    cfg, C, rblocks = shape
    wave = torch.cuda.get_device_properties(0).multi_processor_count // rblocks
    B, t = wave + rest, 0.3
    w = make_weights(cfg, 177, mod_bias_std=0.3)
    r = make_requests(cfg, 178 + rest, B, P, C)
    ex = make_expert(cfg, w, max_batch=B, max_prefix=P, max_chunk=C, max_steps=1)
    try:
        ex.set_prefix_kv(*to_dev_kv(r, cfg))
        v, _ = ex.forward(torch.from_numpy(r["state"]).cuda(), torch.from_numpy(r["noise"]).cuda(), t)
        torch.cuda.synchronize()
        ex.device_status()
    finally:
        ex.close()
    ids = sorted({0, wave - 1, wave, B - 1})
    want, _ = oracle.forward_batch(r["noise"][ids], r["state"][ids], t, r["prefix_k"][:, ids],
                                   r["prefix_v"][:, ids], w, cfg)
    assert_close(v.cpu().numpy()[ids], want, cfg, f"B{B} rest {rest} P{P}")
