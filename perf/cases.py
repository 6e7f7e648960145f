"""Performance cases of the framework: what its users call, over the sizes they call it with.

A program that drives a robot keeps one handle per model and calls, per control cycle: the LLM
prefill of a new observation (``prefill``), the copy of a prefix KV cache made elsewhere
(``prefix``), the future correction module (``correct``), and the flow-matching denoise
(``denoise``). ``layers`` is one expert evaluation of a two-layer expert: the layer stack with its
residual stream as an output. A case is one such call (or the pair compress + predict) on inputs
made from a seed; weights and the handle are made with them.

Weights: N(0, 0.02^2), except the query projection (std 0.06: attention scores of std ~2 instead of
a near-uniform softmax) and the modulation biases (std 0.3: gates large enough that every sublayer
moves the residual stream), as trained weights have them. Prefix keys and values, state, noise and
embeddings are N(0, 1).
"""

from __future__ import annotations

import ctypes
import math
from types import SimpleNamespace

import torch

from paper_2607_12659_gb300 import corr, jpi, prefill

_EXPERT = dict(rope_base=10000.0, rms_eps=1e-6, t_min_period=4e-3, t_max_period=4.0)
MODELS = {
    # The pi0.5 action expert.
    "pi05": dict(n_layers=18, width=1024, n_heads=8, head_dim=256, mlp_dim=4096, action_dim=32, state_dim=32,
                 time_dim=1024, precision="bf16", **_EXPERT),
    # The small fp32 expert.
    "tiny": dict(n_layers=2, width=256, n_heads=4, head_dim=64, mlp_dim=1024, action_dim=7, state_dim=7,
                 time_dim=64, precision="fp32", **_EXPERT),
}
# The Gemma-2B-shaped LLM.
LLM = dict(n_layers=18, width=2048, n_heads=8, head_dim=256, mlp_dim=16384, rope_base=10000.0, rms_eps=1e-6)
# The future correction module at pi0.5 sizes.
CORRECTION = dict(width=1024, n_heads=8, head_dim=128, mlp_dim=2048, d_vlm=2048, n_items=4, action_dim=32,
                  max_delta=50, n_joint=2, ln_eps=1e-6, precision="bf16")


def _expert_shapes(d):
    W, HD, D, F = d.width, d.n_heads * d.head_dim, d.head_dim, d.mlp_dim
    return {
        "state_in_w": (W, d.state_dim), "state_in_b": (W,), "action_in_w": (W, d.action_dim), "action_in_b": (W,),
        "action_out_w": (d.action_dim, W), "action_out_b": (d.action_dim,),
        "time_mlp_in_w": (W, d.time_dim), "time_mlp_in_b": (W,), "time_mlp_out_w": (W, W), "time_mlp_out_b": (W,),
        "final_mod_w": (2 * W, W), "final_mod_b": (2 * W,),
        "wq": (HD, W), "wk": (D, W), "wv": (D, W), "wo": (W, HD),
        "w_gate": (F, W), "w_up": (F, W), "w_down": (W, F),
        "attn_mod_w": (3 * W, W), "attn_mod_b": (3 * W,), "mlp_mod_w": (3 * W, W), "mlp_mod_b": (3 * W,),
    }


def _llm_shapes(d):
    W, HD, D, F = d.width, d.n_heads * d.head_dim, d.head_dim, d.mlp_dim
    return {"attn_norm": (W,), "wq": (HD, W), "wk": (D, W), "wv": (D, W), "wo": (W, HD),
            "mlp_norm": (W,), "w_gate": (F, W), "w_up": (F, W), "w_down": (W, F), "final_norm": (W,)}


def _correction_shapes(d):
    w, f = d.width, d.mlp_dim

    def ln(p):
        return {p + "_w": (w,), p + "_b": (w,)}

    def attn(p, kv):
        return {p + "wq": (w, w), p + "bq": (w,), p + "wk": (w, kv), p + "bk": (w,), p + "wv": (w, kv),
                p + "bv": (w,), p + "wo": (w, w), p + "bo": (w,)}

    def mlp(p):
        return {p + "w1": (f, w), p + "b1": (f,), p + "w2": (w, f), p + "b2": (w,)}

    def block(p):
        return {**ln(p + "ln1"), **attn(p + "sa_", w), **ln(p + "ln2"), **mlp(p + "mlp_")}

    s = {"qf_query": (d.n_items, w), **ln("qf_ln1"), **attn("qf_sa_", w), **ln("qf_ln2"), **attn("qf_ca_", d.d_vlm),
         **ln("qf_ln3"), **mlp("qf_mlp_"), **ln("qf_lnf"), "act_w1": (w, d.action_dim), "act_b1": (w,),
         "act_w2": (w, w), "act_b2": (w,), "act_pos": (d.max_delta, w), **block("ab_"), "fuse_w": (w, 2 * w),
         "fuse_b": (w,)}
    for i in range(d.n_joint):
        s.update(block(f"jb{i}_"))
    s.update({**ln("head_ln"), "corr_w": (w, w), "corr_b": (w,), "conf_w": (1, w), "conf_b": (1,)})
    return s


def listed():
    return [
        # The smallest call: the two-layer fp32 expert of the verification mode.
        {"name": "denoise_tiny_fp32", "kind": "denoise", "model": "tiny", "batch": 1, "prefix": 64, "chunk": 8,
         "steps": 4, "items": 0, "host": False},
        # One Euler step of a short chunk over a short prefix, host buffers in and out: the lowest
        # latency a control loop can ask of the pi0.5 expert.
        {"name": "denoise_b1_short", "kind": "denoise", "model": "pi05", "batch": 1, "prefix": 256, "chunk": 10,
         "steps": 1, "items": 0, "host": True},
        # The headline workload: one robot, three camera images and a text prompt, ten Euler steps.
        {"name": "denoise_b1", "kind": "denoise", "model": "pi05", "batch": 1, "prefix": 816, "chunk": 50,
         "steps": 10, "items": 0, "host": False},
        # A few robots with correction items, an odd prefix length, half the steps.
        {"name": "denoise_b3_items", "kind": "denoise", "model": "pi05", "batch": 3, "prefix": 777, "chunk": 50,
         "steps": 5, "items": 4, "host": False},
        # Batched serving: 8 and 16 requests.
        {"name": "denoise_b8", "kind": "denoise", "model": "pi05", "batch": 8, "prefix": 816, "chunk": 50,
         "steps": 10, "items": 0, "host": False},
        {"name": "denoise_b16", "kind": "denoise", "model": "pi05", "batch": 16, "prefix": 816, "chunk": 50,
         "steps": 10, "items": 0, "host": False},
        # The throughput workload: 64 requests with long multi-view prefixes.
        {"name": "denoise_b64_long", "kind": "denoise", "model": "pi05", "batch": 64, "prefix": 2048, "chunk": 50,
         "steps": 10, "items": 0, "host": False},
        # Two expert layers at a size between them, with the residual stream returned.
        {"name": "layers_b40", "kind": "layers", "model": "pi05", "batch": 40, "prefix": 1333, "chunk": 50,
         "items": 0},
        # The prefix KV cache of one request handed over by another VLM engine.
        {"name": "prefix_b1", "kind": "prefix", "model": "pi05", "batch": 1, "prefix": 816, "fp32": False},
        # The VLM prefill of one observation, all layers.
        {"name": "prefill_b1", "kind": "prefill", "layers": 18, "batch": 1, "prefix": 816, "fp32": False},
        # Four LLM layers over a batch of odd-length prefixes.
        {"name": "prefill_b4_layers", "kind": "prefill", "layers": 4, "batch": 4, "prefix": 1037, "fp32": True},
        # The future correction module after a fresh VLM output: compress, then predict 9 actions ahead.
        {"name": "correct_b1", "kind": "correct", "batch": 1, "tokens": 816, "delta": 9, "fp32": False},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["denoise", "denoise", "denoise", "layers", "prefix", "prefill", "correct"])
    prefix = _log(rng, 64, 2048)
    if kind == "denoise":
        model = "tiny" if rng.random() < 0.15 else "pi05"
        batch = _log(rng, 1, 4) if model == "tiny" else _log(rng, 1, 64)
        return {"kind": kind, "model": model, "batch": batch, "prefix": prefix, "chunk": rng.randint(4, 50),
                "steps": rng.randint(1, 10), "items": rng.choice([0, 0, 4]), "host": rng.random() < 0.3}
    if kind == "layers":
        return {"kind": kind, "model": "pi05", "batch": _log(rng, 1, 64), "prefix": prefix,
                "chunk": rng.randint(4, 50), "items": rng.choice([0, 0, 4])}
    if kind == "prefix":
        return {"kind": kind, "model": "pi05", "batch": _log(rng, 1, 64), "prefix": prefix,
                "fp32": rng.random() < 0.3}
    if kind == "prefill":
        return {"kind": kind, "layers": rng.randint(1, 6), "batch": _log(rng, 1, 8), "prefix": _log(rng, 64, 1536),
                "fp32": rng.random() < 0.3}
    return {"kind": kind, "batch": _log(rng, 1, 16), "tokens": _log(rng, 64, 2048), "delta": _log(rng, 1, 50),
            "fp32": rng.random() < 0.5}


# ------------------------------------------------------------------ inputs

class _Handle:
    """A library handle that is destroyed with the state that holds it."""

    def __init__(self, raw, destroy):
        self.raw, self._destroy = raw, destroy

    def __del__(self):
        try:
            self._destroy(self.raw)
        except Exception:
            pass


class _Draw:
    def __init__(self, seed):
        self.g = torch.Generator(device="cuda")
        self.g.manual_seed(int(seed))

    def __call__(self, *shape, std=1.0, bf16=False):
        x = torch.randn(shape, generator=self.g, device="cuda", dtype=torch.float32) * std
        return x.to(torch.bfloat16).float() if bf16 else x


def _expert_dims(case):
    d = SimpleNamespace(**MODELS[case["model"]])
    if case["kind"] == "layers":
        d.n_layers = 2
    return d


def _llm_dims(case):
    return SimpleNamespace(**dict(LLM, n_layers=case["layers"]))


def _expert_weights(dims, rnd):
    """Device fp32 tensors by name (per-layer lists); in bf16 precision the matrices hold bf16 values."""
    shapes, bf16 = _expert_shapes(dims), dims.precision == "bf16"

    def one(name):
        if len(shapes[name]) == 2:
            return rnd(*shapes[name], std=0.06 if name == "wq" else 0.02, bf16=bf16)
        return rnd(*shapes[name], std=0.3 if name.endswith("mod_b") else 0.02)

    w = {n: one(n) for n in jpi.GLOBAL_WEIGHTS}
    w.update({n: [one(n) for _ in range(dims.n_layers)] for n in jpi.LAYER_WEIGHTS})
    return w


def _expert_handle(dims, w, batch, prefix, chunk, steps):
    wt = jpi.jpi_weights(on_device=1)
    for n in jpi.GLOBAL_WEIGHTS:
        setattr(wt, n, w[n].data_ptr())
    tabs = []
    for n in jpi.LAYER_WEIGHTS:
        tabs.append((ctypes.c_void_p * dims.n_layers)(*[t.data_ptr() for t in w[n]]))
        setattr(wt, n, ctypes.cast(tabs[-1], ctypes.c_void_p))
    torch.cuda.synchronize()
    cfg = jpi.make_config(dims, batch, prefix, chunk, steps)
    return _Handle(jpi.jpi_expert_create(cfg, wt), jpi.jpi_expert_destroy)


def _expert_inputs(case, seed):
    dims, rnd = _expert_dims(case), _Draw(seed)
    bf16 = dims.precision == "bf16"
    B, P, C, T = case["batch"], case["prefix"], case.get("chunk", 1), case.get("items", 0)
    s = {"dims": dims, "w": _expert_weights(dims, rnd) if case["kind"] != "prefix" else None}
    s["k"], s["v"] = rnd(dims.n_layers, B, P, dims.head_dim), rnd(dims.n_layers, B, P, dims.head_dim)
    if bf16 and not case.get("fp32"):
        s["k"], s["v"] = s["k"].to(torch.bfloat16), s["v"].to(torch.bfloat16)
    s["state"], s["noise"] = rnd(B, dims.state_dim), rnd(B, C, dims.action_dim)
    s["items"] = rnd(B, T, dims.width, std=0.5) if T else None
    return s


def _llm_inputs(case, seed):
    dims, rnd = _llm_dims(case), _Draw(seed)
    shapes = _llm_shapes(dims)

    def one(name):
        if len(shapes[name]) == 2:
            return rnd(*shapes[name], std=0.02, bf16=True)
        return rnd(*shapes[name], std=0.1)

    w = {n: [one(n) for _ in range(dims.n_layers)] for n in prefill.LAYER_WEIGHTS}
    w["final_norm"] = one("final_norm")
    x = rnd(case["batch"], case["prefix"], dims.width)
    return {"dims": dims, "w": w, "x": x if case["fp32"] else x.to(torch.bfloat16)}


def _correct_inputs(case, seed):
    dims, rnd = SimpleNamespace(**CORRECTION), _Draw(seed)
    w = {}
    for name, shape in _correction_shapes(dims).items():
        if len(shape) == 2:
            w[name] = rnd(*shape, std=0.02, bf16=True)
        else:
            w[name] = rnd(*shape, std=0.1) + 1.0 if name.endswith("_w") and "ln" in name else rnd(*shape, std=0.02)
    hv = rnd(case["batch"], case["tokens"], dims.d_vlm)
    return {"dims": dims, "w": w, "h_vlm": hv if case["fp32"] else hv.to(torch.bfloat16),
            "actions": rnd(case["batch"], case["delta"], dims.action_dim)}


class _KvView:
    """A [B][rows][D] view of one layer's K or V in the handle's store, for torch.as_tensor; it
    keeps the handle, and so the store, alive."""

    def __init__(self, handle, ptr, batch, rows, dim, stride):
        self.handle = handle
        # bf16 has no interface code: 16-bit integers carry the same bits.
        self.__cuda_array_interface__ = {"shape": (batch, rows, dim), "typestr": "<i2", "version": 3,
                                         "strides": (stride * 2, dim * 2, 2), "data": (ptr, False)}


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("denoise", "layers"):
        s = _expert_inputs(case, seed)
        dims, B, P, C = s["dims"], case["batch"], case["prefix"], case["chunk"]
        s["h"] = _expert_handle(dims, s.pop("w"), B, P, C, case.get("steps", 1))
        jpi.jpi_set_prefix_kv(s["h"].raw, list(s["k"]), list(s["v"]), B, P, s["k"].dtype == torch.float32)
        if s["items"] is not None:
            jpi.jpi_set_correction(s["h"].raw, s["items"], B, case["items"])
        if kind == "layers":
            S = 1 + case["items"] + C
            s["hidden"] = torch.empty((B, S, dims.width), dtype=torch.float32, device="cuda")
        if case.get("host"):
            s["state"], s["noise"] = s["state"].cpu().pin_memory(), s["noise"].cpu().pin_memory()
            s["out"] = torch.empty_like(s["noise"]).pin_memory()
        else:
            s["out"] = torch.empty_like(s["noise"])
        torch.cuda.synchronize()
        del s["k"], s["v"]
    elif kind == "prefix":
        s = _expert_inputs(case, seed)
        dims, B, P = s["dims"], case["batch"], case["prefix"]
        # The store's size is the layer geometry's; the weights play no part in this call.
        small = SimpleNamespace(**dict(vars(dims), width=128, mlp_dim=64, time_dim=64))
        s["h"] = _expert_handle(small, _expert_weights(small, _Draw(seed)), B, P, 50, 1)
        s["k"], s["v"], s["store"] = list(s["k"]), list(s["v"]), []
        for l in range(dims.n_layers):
            k, v, stride = jpi.jpi_prefix_kv_ptr(s["h"].raw, l)
            for p in (k, v):
                view = torch.as_tensor(_KvView(s["h"], p, B, P, dims.head_dim, stride), device="cuda")
                s["store"].append(view.view(torch.bfloat16))
                s["store"][-1].owner = s["h"]
    elif kind == "prefill":
        s = _llm_inputs(case, seed)
        dims, w = s["dims"], s.pop("w")
        wt, tabs = prefill.jpi_prefill_weights(on_device=1), []
        for n in prefill.LAYER_WEIGHTS:
            tabs.append((ctypes.c_void_p * dims.n_layers)(*[t.data_ptr() for t in w[n]]))
            setattr(wt, n, ctypes.cast(tabs[-1], ctypes.c_void_p))
        wt.final_norm = w["final_norm"].data_ptr()
        torch.cuda.synchronize()
        s["h"] = _Handle(prefill.jpi_prefill_create(
            prefill.make_prefill_config(dims, case["batch"], case["prefix"]), wt), prefill.jpi_prefill_destroy)
        shape = (dims.n_layers, case["batch"], case["prefix"], dims.head_dim)
        s["k"] = torch.empty(shape, dtype=torch.bfloat16, device="cuda")
        s["v"] = torch.empty(shape, dtype=torch.bfloat16, device="cuda")
        s["kp"], s["vp"] = ([t[l].data_ptr() for l in range(dims.n_layers)] for t in (s["k"], s["v"]))
        s["final"] = torch.empty(s["x"].shape, dtype=torch.float32, device="cuda")
    else:
        s = _correct_inputs(case, seed)
        w = {n: t.cpu().numpy() for n, t in s.pop("w").items()}
        s["h"] = corr.Corrector(s["dims"], w, max_batch=case["batch"], max_vlm_tokens=case["tokens"])
    s["case"] = dict(case)
    return s


def run(s):
    c = s["case"]
    if c["kind"] == "denoise":
        call = jpi.jpi_denoise_host if c["host"] else jpi.jpi_denoise
        call(s["h"].raw, s["state"], s["noise"], c["batch"], c["chunk"], c["steps"], s["out"])
        return s["out"]
    if c["kind"] == "layers":
        jpi.jpi_expert_forward(s["h"].raw, s["state"], s["noise"], 0.3, c["batch"], c["chunk"], s["out"], s["hidden"])
        return {"v": s["out"], "h": s["hidden"]}
    if c["kind"] == "prefix":
        jpi.jpi_set_prefix_kv(s["h"].raw, s["k"], s["v"], c["batch"], c["prefix"], c["fp32"])
        return s["store"]
    if c["kind"] == "prefill":
        B, P = c["batch"], c["prefix"]
        prefill.jpi_prefill_run(s["h"].raw, s["x"], c["fp32"], B, P, s["kp"], s["vp"], P * s["dims"].head_dim, s["final"])
        return {"k": s["k"], "v": s["v"], "final": s["final"]}
    z = s["h"].compress(s["h_vlm"])
    pred, conf = s["h"].predict(z, s["actions"])
    return {"state": z, "predicted": pred, "confidence": conf}


# ------------------------------------------------------------------ work

def work(case):
    kind = case["kind"]
    if kind in ("denoise", "layers", "prefix"):
        d = _expert_dims(case)
        B, P, L, D, H, W, F = case["batch"], case["prefix"], d.n_layers, d.head_dim, d.n_heads, d.width, d.mlp_dim
        e = 2 if d.precision == "bf16" else 4
        kv = 2 * L * B * P * D
        if kind == "prefix":
            return {"bytes": kv * ((4 if case["fp32"] else 2) + e), "flops": 0}
        N, C = case.get("steps", 1), case["chunk"]
        S = 1 + case["items"] + C
        proj = W * (H + 2) * D + H * D * W + 3 * W * F
        mods = (6 * L + 2) * W * W + W * d.time_dim + W * W
        io = 4 * B * (d.state_dim + 2 * C * d.action_dim + (S * W if kind == "layers" else 0))
        # The layers' weights (623 MB at pi0.5 sizes) fit no on-chip memory: every Euler step reads
        # them again. The modulation weights and the prefix KV count once.
        if L * proj * e < 100e6:
            weights = (L * proj + mods) * e
        else:
            weights = (N * L * proj + mods) * e
        flops = 2.0 * N * B * S * (L * (proj + 2 * H * D * (P + S)) + 2 * W * d.action_dim) + 2.0 * N * mods
        return {"bytes": weights + kv * e + io, "flops": flops}
    if kind == "prefill":
        d = _llm_dims(case)
        L, D, H, W, F, B, P = d.n_layers, d.head_dim, d.n_heads, d.width, d.mlp_dim, case["batch"], case["prefix"]
        proj = W * (H + 2) * D + H * D * W + 3 * W * F
        M = B * P
        return {"bytes": 2 * L * proj + M * W * ((4 if case["fp32"] else 2) + 4) + 2 * L * M * D * 2,
                "flops": 2.0 * L * M * (proj + 2 * H * D * P)}
    d = SimpleNamespace(**CORRECTION)
    B, T, n = case["batch"], case["tokens"], case["delta"]
    w, f = d.width, d.mlp_dim
    blk = 4 * w * w + 2 * w * f                       # q, k, v, o, MLP
    comp = w * d.d_vlm + w * w + 2 * w * f            # value map, output projection, MLP (queries are fixed)
    pred = w * d.action_dim + w * w + (d.n_joint + 1) * blk + 2 * w * w + w * w
    qk = d.n_heads * d.n_items * d.d_vlm
    vlm = B * T * d.d_vlm
    rows = B * d.n_items
    flops = 2.0 * (2 * vlm * d.n_heads * d.n_items + rows * comp + B * n * (w * d.action_dim + 3 * w * w)
                   + rows * (d.n_joint * blk + 3 * w * w) + B * (2 * w * w + 2 * w * f))
    return {"bytes": 2 * (comp + pred) + 4 * qk + vlm * (4 if case["fp32"] else 2) + 4 * B * n * d.action_dim
            + 4 * 2 * rows * w, "flops": flops}


def tolerance(case):
    kind = case["kind"]
    if kind == "prefix":
        return "exact"      # a copy, or a rounding to bf16
    # About four times the error against the 64-bit results, measured: 1e-7 in fp32; with bf16
    # operands 4e-3 (ten steps) to 9e-3 (one step) for the actions, 4e-3 for two layers, 2e-3 to
    # 1.1e-2 for the prefill's output (growing with the layers); 3e-7 to 8e-7 (the confidence, one
    # value per request) in the correction module, whose activations and sums are fp32.
    if kind == "denoise":
        return {"rel": 2e-6} if case["model"] == "tiny" else {"rel": 3e-2}
    if kind == "prefill":
        return {"rel": 3e-2}
    return {"rel": 2e-2 if kind == "layers" else 5e-6}


# ------------------------------------------------------------------ 64-bit results

F8 = torch.float64


def _rope(x, pos, base):
    half = x.shape[-1] // 2
    ang = pos.to(F8)[:, None] * base ** (-2.0 * torch.arange(half, device=x.device, dtype=F8) / x.shape[-1])
    shape = (1, len(pos)) + (1,) * (x.dim() - 3) + (half,)
    cos, sin = ang.cos().reshape(shape), ang.sin().reshape(shape)
    a, b = x[..., :half], x[..., half:]
    return torch.cat([a * cos - b * sin, b * cos + a * sin], -1)


def _gelu(y):
    return 0.5 * y * (1 + torch.tanh(math.sqrt(2 / math.pi) * (y + 0.044715 * y ** 3)))


def _attend(q, k, v, hidden=None):
    """q [B][S][H][D] against k, v [B][K][D]; hidden [S][K]: keys a row does not see."""
    B, S, H, D = q.shape
    s = (q.reshape(B, S * H, D) @ k.transpose(1, 2) / math.sqrt(D)).reshape(B, S, H, -1)
    if hidden is not None:
        s = s.masked_fill(hidden[None, :, None, :], -math.inf)
    return (s.softmax(-1).reshape(B, S * H, -1) @ v).reshape(B, S, H * D)


def _forward64(x, state, items, t, pk, pv, w, d):
    B, C, _ = x.shape
    ctx = 1 + (0 if items is None else items.shape[1])
    P, S, W, H, D = pk.shape[2], ctx + C, d.width, d.n_heads, d.head_dim
    half = d.time_dim // 2
    period = d.t_min_period * (d.t_max_period / d.t_min_period) ** (
        torch.arange(half, device=x.device, dtype=F8) / (half - 1))
    e = torch.cat([torch.sin(2 * math.pi * t / period), torch.cos(2 * math.pi * t / period)])
    silu = torch.nn.functional.silu
    c = silu(w["time_mlp_in_w"].double() @ e + w["time_mlp_in_b"].double())
    c = silu(w["time_mlp_out_w"].double() @ c + w["time_mlp_out_b"].double())

    def norm(h, sg, be):
        return h / torch.sqrt((h * h).mean(-1, keepdim=True) + d.rms_eps) * (1 + sg) + be

    parts = [(state @ w["state_in_w"].double().T + w["state_in_b"].double())[:, None]]
    if items is not None:
        parts.append(items)
    parts.append(x @ w["action_in_w"].double().T + w["action_in_b"].double())
    h = torch.cat(parts, 1)
    hidden = torch.zeros((S, P + S), dtype=torch.bool, device=x.device)
    hidden[:ctx, P + ctx:] = True
    pos = P + torch.arange(S, device=x.device)
    for l in range(d.n_layers):
        m = lambda n: w[n][l].double()  # noqa: E731
        ma, mm = m("attn_mod_w") @ c + m("attn_mod_b"), m("mlp_mod_w") @ c + m("mlp_mod_b")
        u = norm(h, ma[:W], ma[W:2 * W])
        q = _rope((u @ m("wq").T).reshape(B, S, H, D), pos, d.rope_base)
        k = _rope(u @ m("wk").T, pos, d.rope_base)
        o = _attend(q, torch.cat([pk[l].double(), k], 1), torch.cat([pv[l].double(), u @ m("wv").T], 1), hidden)
        h = h + ma[2 * W:] * (o @ m("wo").T)
        u = norm(h, mm[:W], mm[W:2 * W])
        h = h + mm[2 * W:] * ((_gelu(u @ m("w_gate").T) * (u @ m("w_up").T)) @ m("w_down").T)
    fm = w["final_mod_w"].double() @ c + w["final_mod_b"].double()
    return norm(h, fm[:W], fm[W:])[:, ctx:] @ w["action_out_w"].double().T + w["action_out_b"].double(), h


def _ln64(x, w, b, eps):
    mu = x.mean(-1, keepdim=True)
    return (x - mu) / torch.sqrt(((x - mu) ** 2).mean(-1, keepdim=True) + eps) * w + b


def _mha64(xq, xkv, w, p, d):
    q, k, v = (x @ w[p + "w" + n].T + w[p + "b" + n] for x, n in ((xq, "q"), (xkv, "k"), (xkv, "v")))
    q, k, v = (t.reshape(t.shape[0], t.shape[1], d.n_heads, d.head_dim).transpose(1, 2) for t in (q, k, v))
    o = (q @ k.transpose(2, 3) / math.sqrt(d.head_dim)).softmax(-1) @ v
    return o.transpose(1, 2).reshape(xq.shape[0], xq.shape[1], -1) @ w[p + "wo"].T + w[p + "bo"]


def _block64(x, w, p, d):
    u = _ln64(x, w[p + "ln1_w"], w[p + "ln1_b"], d.ln_eps)
    x = x + _mha64(u, u, w, p + "sa_", d)
    u = _ln64(x, w[p + "ln2_w"], w[p + "ln2_b"], d.ln_eps)
    return x + _gelu(u @ w[p + "mlp_w1"].T + w[p + "mlp_b1"]) @ w[p + "mlp_w2"].T + w[p + "mlp_b2"]


def exact(case, seed):
    kind = case["kind"]
    if work(case)["flops"] > 1e13:
        return None         # over about 20 seconds in 64 bits
    if kind == "prefix":
        s = _expert_inputs(case, seed)
        return [t for l in range(s["dims"].n_layers) for t in (s["k"][l].to(torch.bfloat16), s["v"][l].to(torch.bfloat16))]
    if kind in ("denoise", "layers"):
        s = _expert_inputs(case, seed)
        items = None if s["items"] is None else s["items"].double()
        args = (s["k"], s["v"], s["w"], s["dims"])
        if kind == "layers":
            v, h = _forward64(s["noise"].double(), s["state"].double(), items, float(torch.tensor(0.3)), *args)
            return {"v": v, "h": h}
        x, N = s["noise"].double(), case["steps"]
        for n in range(N):
            x = x + _forward64(x, s["state"].double(), items, n / N, *args)[0] / N
        return x.cpu() if case["host"] else x
    if kind == "prefill":
        s = _llm_inputs(case, seed)
        d, w, h = s["dims"], s["w"], s["x"].double()
        B, P, W = h.shape
        pos = torch.arange(P, device=h.device)
        norm = lambda x, a: x / torch.sqrt((x * x).mean(-1, keepdim=True) + d.rms_eps) * (1 + a.double())  # noqa: E731
        ks, vs = [], []
        for l in range(d.n_layers):
            m = lambda n: w[n][l].double()  # noqa: E731
            u = norm(h, w["attn_norm"][l])
            q = _rope((u @ m("wq").T).reshape(B, P, d.n_heads, d.head_dim), pos, d.rope_base)
            k, v = _rope(u @ m("wk").T, pos, d.rope_base), u @ m("wv").T
            ks.append(k)
            vs.append(v)
            h = h + _attend(q, k, v) @ m("wo").T
            u = norm(h, w["mlp_norm"][l])
            h = h + (_gelu(u @ m("w_gate").T) * (u @ m("w_up").T)) @ m("w_down").T
        return {"k": torch.stack(ks), "v": torch.stack(vs), "final": norm(h, w["final_norm"])}
    s = _correct_inputs(case, seed)
    d, w = s["dims"], {n: t.double() for n, t in s["w"].items()}
    B, n = case["batch"], case["delta"]
    hv = s["h_vlm"].double()
    x = w["qf_query"][None].expand(B, -1, -1)
    u = _ln64(x, w["qf_ln1_w"], w["qf_ln1_b"], d.ln_eps)
    x = x + _mha64(u, u, w, "qf_sa_", d)
    u = _ln64(x, w["qf_ln2_w"], w["qf_ln2_b"], d.ln_eps)
    x = x + _mha64(u, hv, w, "qf_ca_", d)
    u = _ln64(x, w["qf_ln3_w"], w["qf_ln3_b"], d.ln_eps)
    x = x + _gelu(u @ w["qf_mlp_w1"].T + w["qf_mlp_b1"]) @ w["qf_mlp_w2"].T + w["qf_mlp_b2"]
    z = _ln64(x, w["qf_lnf_w"], w["qf_lnf_b"], d.ln_eps)
    a = _gelu(s["actions"].double() @ w["act_w1"].T + w["act_b1"]) @ w["act_w2"].T + w["act_b2"] + w["act_pos"][:n]
    last = _block64(a, w, "ab_", d)[:, -1:]
    x = torch.cat([z, last.expand(-1, z.shape[1], -1)], -1) @ w["fuse_w"].T + w["fuse_b"]
    for i in range(d.n_joint):
        x = _block64(x, w, f"jb{i}_", d)
    u = _ln64(x, w["head_ln_w"], w["head_ln_b"], d.ln_eps)
    return {"state": z, "predicted": u @ w["corr_w"].T + w["corr_b"],
            "confidence": u.mean(1) @ w["conf_w"][0] + w["conf_b"][0]}
