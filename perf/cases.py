"""The work that users of this library have it do, as cases with inputs, one pass and a bound on its cost.

A case is a dict of plain values.  Kinds:

  layer    one mixer layer on a batch of sequences: gate from the pooled queries, spectral mixing of the values,
           and on patch grids the Haar refinement
  project  the same layer entered with the hidden states: Q/V projections (whose query sum feeds the gate) first
  train    a layer's forward pass and the gradients of the mixing with respect to the values and the gate
  prompt   the start of a generation: prefill of the Prefix-FFT cache from a prompt shorter than the window, the gate of
           the running query sum, and the mixed rows of the prompt read back from the cached spectrum
  decode   one token of a generation: cache update, gate, read-out of the newest rows; the position advances with each pass
  append   one token taken into the cache without reading anything out

All heads are 64 channels wide and all gate networks have 64 hidden units, as in the workloads of
paper_2502_18394_b200/workloads.py; gate weights follow its recipe too (std 0.02).
"""
import math

import torch

from paper_2502_18394_b200 import binding as S

D = 64
HIDDEN = 64
DTYPES = {"f32": torch.float32, "bf16": torch.bfloat16, "f16": torch.float16}
SIZE = {"f32": 4, "bf16": 2, "f16": 2}
POOL = 32                                                  # tokens that a decoding loop cycles through


def _layer(B, L, H, n, dtype, toeplitz=0, levels=0, kind="layer"):
    return {"kind": kind, "B": B, "L": L, "H": H, "n": n, "dtype": dtype, "toeplitz": toeplitz, "levels": levels}


def _cache(kind, B, L, H, n, dtype, rows=0):
    return {"kind": kind, "B": B, "L": L, "H": H, "n": n, "dtype": dtype, "rows": rows}


def listed():
    return [
        # the smallest call: one 1k sequence, two heads, fp32; launches and host time count
        dict(_layer(1, 1024, 2, 1024, "f32"), name="layer_1k_f32"),
        # the 8k and 128k contexts of the paper's throughput figure
        dict(_layer(1, 8192, 32, 8192, "bf16"), name="layer_8k_bf16"),
        dict(_layer(1, 131072, 32, 131072, "bf16"), name="layer_128k_bf16"),
        # an image batch: 14 x 14 patches, refinement of two levels
        dict(_layer(256, 196, 12, 196, "bf16", levels=2), name="layer_vit_bf16"),
        # a batch of prompts of no convenient length, zero-padded to the next power of two, banded gate update
        dict(_layer(4, 5003, 12, 8192, "f16", toeplitz=2), name="layer_ragged_f16"),
        # hidden states in, four sequences of 4k
        dict(_layer(4, 4096, 16, 4096, "bf16", kind="project"), name="project_4k_bf16"),
        # training at a 1k context (batch of 16) and at 8k
        dict(_layer(16, 1024, 12, 1024, "bf16", kind="train"), name="train_1k_bf16"),
        dict(_layer(1, 8192, 32, 8192, "bf16", kind="train"), name="train_8k_bf16"),
        # two prompts of some 20k tokens into the 32k window
        dict(_cache("prompt", 2, 20011, 32, 32768, "bf16"), name="prompt_32k_bf16"),
        # one user with a short window: latency of a token
        dict(_cache("decode", 1, 2500, 12, 4096, "f16", rows=1), name="decode_4k_f16"),
        # eight users with the 32k window: the whole step, and the update alone
        dict(_cache("decode", 8, 20011, 32, 32768, "bf16", rows=1), name="decode_32k_bf16"),
        dict(_cache("append", 8, 20011, 32, 32768, "bf16"), name="append_32k_bf16"),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _pow2(rng, lo, hi):
    return 1 << rng.randint(int(math.log2(lo)), int(math.log2(hi)))


def _batch(rng, H, n, most):
    """Sequences of n tokens with H heads that keep B H n D under `most` elements."""
    return _log_int(rng, 1, max(1, min(256, most // (H * n * D))))


def draw(rng):
    kind = rng.choice(["layer", "layer", "layer", "project", "train", "prompt", "decode", "append"])
    H = rng.choice([2, 4, 8, 12, 16, 32])
    dtype = rng.choice(["bf16", "bf16", "f16", "f32"])
    if kind == "layer":
        what = rng.choice(["power", "ragged", "grid"])
        toeplitz = rng.choice([0, 0, 2])
        if what == "grid":                                 # square patch grids
            L = rng.choice([14, 16, 20, 24, 28, 32]) ** 2
            return _layer(_batch(rng, H, L, 1 << 26), L, H, L, dtype, toeplitz, rng.choice([0, 1, 2]))
        n = _pow2(rng, 512, 131072)
        L = n if what == "power" else rng.randint(n // 2 + 1, n)
        H = min(H, 8) if n > 32768 else H
        return _layer(_batch(rng, H, n, 1 << 26), L, H, n, dtype, toeplitz)
    if kind == "project":
        n = _pow2(rng, 1024, 32768)
        L = rng.choice([n, rng.randint(n // 2 + 1, n)])
        return _layer(_batch(rng, H, n, 1 << 25), L, H, n, "bf16", kind="project")
    if kind == "train":
        n = _pow2(rng, 512, 32768)
        L = rng.choice([n, rng.randint(n // 2 + 1, n)])
        return _layer(_batch(rng, H, n, 1 << 25), L, H, n, dtype, kind="train")
    n = _pow2(rng, 1024, 32768)
    L = rng.randint(n // 4, n)
    B = min(8, _batch(rng, H, n, 1 << 26))
    return _cache(kind, B, L, H, n, dtype, rows=rng.randint(1, 4) if kind == "decode" else 0)


_contexts = {}


def _context():
    """A program keeps one context per device."""
    d = torch.cuda.current_device()
    if d not in _contexts:
        _contexts[d] = S.Context(d)
    return _contexts[d]


class _Inputs:
    def __init__(self, seed):
        self.gen = torch.Generator(device="cuda")
        self.gen.manual_seed(seed)

    def normal(self, shape, std=1.0, dtype=torch.float32):
        return (torch.randn(shape, generator=self.gen, device="cuda", dtype=torch.float32) * std).to(dtype)

    def tokens(self, B, L, H, dtype):
        """Token features: unit variance around a per-channel offset."""
        x = torch.randn((B, L, H, D), generator=self.gen, device="cuda", dtype=torch.float32)
        return x.add_(0.5 * torch.randn((1, 1, H, D), generator=self.gen, device="cuda")).to(dtype)

    def gate(self, H, n, dtype, toeplitz=0):
        wd = torch.float32 if dtype == "f32" else torch.bfloat16
        K = n // 2 + 1
        return {
            "ln_gamma": 1.0 + self.normal((H, D), 0.1), "ln_beta": self.normal((H, D), 0.1), "ln_eps": 1e-5,
            "W1": self.normal((H, D, HIDDEN), 0.02, wd), "b1": self.normal((H, HIDDEN), 0.02),
            "W2": self.normal((H, HIDDEN, 2 * K), 0.02, wd), "b2": self.normal((H, 2 * K), 0.02), "hidden": HIDDEN,
            "modrelu_bias": self.normal((H, K), 0.002),
            "toeplitz": self.normal((H, 2 * toeplitz + 1, 2), 0.1) if toeplitz else None,
        }

    def refinement(self, B, H, levels):
        return {
            "Ww1": self.normal((H, D, HIDDEN), 0.02, torch.bfloat16), "bw1": self.normal((H, HIDDEN), 0.02),
            "Ww2": self.normal((H, HIDDEN, (levels + 1) * D), 0.02, torch.bfloat16),
            "bw2": self.normal((H, (levels + 1) * D), 0.02), "hidden": HIDDEN, "levels": levels,
            "qbar": torch.empty((B, H, D), device="cuda"),
        }


def prepare(case, seed):
    x = _Inputs(seed)
    B, L, H, n, dt = case["B"], case["L"], case["H"], case["n"], DTYPES[case["dtype"]]
    s = {"kind": case["kind"], "ctx": _context(), "n": n}
    s["gate"] = x.gate(H, n, case["dtype"], case.get("toeplitz", 0)) if case["kind"] != "append" else None
    if case["kind"] == "project":
        s["x"] = x.tokens(B, L, H, dt)
        s["Wq"], s["Wv"] = (x.normal((H, D, D), D ** -0.5, dt) for _ in range(2))
        return s
    if case["kind"] in ("layer", "train"):
        s["q"], s["v"] = x.tokens(B, L, H, dt), x.tokens(B, L, H, dt)
        s["wrm"] = x.refinement(B, H, case["levels"]) if case["levels"] else None
        if case["kind"] == "train":
            s["dy"] = x.normal((B, L, H, D), 1.0, dt)
        return s
    cache = S.PrefixCache(B, H, D, n, dtype=dt)
    s["cache"] = cache
    q, v = x.tokens(B, L, H, dt), x.tokens(B, L, H, dt)
    if case["kind"] == "prompt":
        s["q"], s["v"], s["L"] = q, v, L
        return s
    # a generation in progress: the cache holds the prompt, the loop keeps its buffers
    S.spectre_prefix_cache_prefill(s["ctx"], cache, q, v)
    s["q_t"], s["v_t"], s["t"] = x.tokens(POOL, B, H, dt), x.tokens(POOL, B, H, dt), L
    if case["kind"] == "decode":
        s["rows"] = list(range(n - case["rows"], n))
        s["y"] = torch.empty((B, case["rows"], H, D), dtype=dt, device="cuda")
        s["g"] = torch.empty((B, H, n // 2 + 1, 2), device="cuda")
        need = S.spectre_decode_workspace_bytes(s["ctx"], B, H, D, n, case["rows"])
        s["ws"] = torch.empty(max(need, 16), dtype=torch.uint8, device="cuda")
    return s


def _state(cache):
    return {"spectrum": cache.prefix_fft, "V": cache.V_buf, "Q": cache.Q_buf, "sum_q": cache.sum_q}


def run(s):
    ctx, kind, n = s["ctx"], s["kind"], s["n"]
    if kind == "layer":
        wrm = s["wrm"]
        g = S.spectre_gate(ctx, s["gate"], n, q=s["q"], qbar_out=wrm["qbar"] if wrm else None)
        return {"g": g, "y": S.spectre_mixer_forward(ctx, s["v"], g, n_fft=n, wrm=wrm)}
    if kind == "project":
        q, v, sum_q = S.spectre_project_qv(ctx, s["x"], s["Wq"], s["Wv"])
        g = S.spectre_gate(ctx, s["gate"], n, sum_q=sum_q, inv_count=1.0 / v.shape[1])
        return {"q": q, "v": v, "sum_q": sum_q, "g": g, "y": S.spectre_mixer_forward(ctx, v, g, n_fft=n)}
    if kind == "train":
        g = S.spectre_gate(ctx, s["gate"], n, q=s["q"])
        y = S.spectre_mixer_forward(ctx, s["v"], g, n_fft=n)
        dv, dg = S.spectre_mixer_backward(ctx, s["v"], s["dy"], g, n_fft=n)
        return {"g": g, "y": y, "dv": dv, "dg": dg}
    cache = s["cache"]
    if kind == "prompt":
        S.spectre_prefix_cache_prefill(ctx, cache, s["q"], s["v"])
        g = S.spectre_gate(ctx, s["gate"], n, sum_q=cache.sum_q, inv_count=1.0 / n)
        y = torch.empty_like(s["v"])
        return dict(_state(cache), g=g, y=S.spectre_prefix_cache_readout(ctx, cache, g, y=y))
    t = s["t"]
    s["t"] = t + 1
    q_t, v_t = s["q_t"][t % POOL], s["v_t"][t % POOL]
    if kind == "append":
        S.spectre_prefix_cache_append(ctx, cache, q_t, v_t, t)
        return _state(cache)
    y, g = S.spectre_prefix_cache_decode_step(ctx, cache, q_t, v_t, t, s["gate"], s["rows"], y_rows=s["y"], g_out=s["g"],
                                              workspace=s["ws"])
    return dict(_state(cache), g=g, y=y)


def work(case):
    B, L, H, n, es = case["B"], case["L"], case["H"], case["n"], SIZE[case["dtype"]]
    K = n // 2 + 1
    act = es * B * L * H * D                                # one [B, L, H, D] tensor
    spectrum = 8.0 * B * H * K * D
    fft = 2.5 * B * H * D * n * max(1.0, math.log2(n))      # one real transform of every column
    ws = 4 if case["dtype"] == "f32" else 2
    gate_bytes = H * (ws * HIDDEN * (D + 2 * K) + 4 * 3 * K) + 8.0 * B * H * K   # weights in, gate out
    gate_flops = 2.0 * B * H * HIDDEN * (D + 2 * K)
    kind = case["kind"]
    if kind == "layer":                                     # q, v in, y out
        return {"bytes": 3 * act + gate_bytes, "flops": act / es + 2 * fft + gate_flops}
    if kind == "project":                                   # x in, q, v, y out
        return {"bytes": 4 * act + gate_bytes, "flops": 4.0 * act / es * D + 2 * fft + gate_flops}
    if kind == "train":                                     # q, v, dy in, y, dv out, the gate's gradient
        return {"bytes": 5 * act + gate_bytes + 8.0 * B * H * K, "flops": act / es + 4 * fft + gate_flops + 8.0 * B * H * K * D}
    ring = es * B * n * H * D                               # one ring buffer
    if kind == "prompt":                                    # q, v in; spectrum, both rings and y out
        return {"bytes": 3 * act + 2 * ring + spectrum + gate_bytes, "flops": act / es + 2 * fft + gate_flops}
    token = 8.0 * B * H * K * D                             # a complex multiply-add of one real number per bin and channel
    if kind == "append":                                    # the spectrum in and out
        return {"bytes": 2 * spectrum + 4 * es * B * H * D, "flops": token}
    return {"bytes": 2 * spectrum + gate_bytes + 4 * es * B * H * D, "flops": token * (1 + case["rows"]) + gate_flops}


def tolerance(case):
    if case["kind"] == "append" or case["dtype"] == "f32":  # fp32 spectra, fp32 transforms
        return {"rel": 2e-5}
    # 16-bit rows; the tensor-core transforms keep fp16 operands between their stages
    return {"rel": 5e-3 if case["dtype"] == "bf16" else 3e-3}
