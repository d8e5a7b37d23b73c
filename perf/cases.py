"""Performance cases of the ATP prefill path: what a program that uses this library has it do.

A case is one call pattern of the public binding at one size:

  layer        one AtpLayer.forward: Norm -> principal basis -> attention on r principal keys, and, where the layer
               has them, output projection and FeedForward through the low-rank representation
  basis        the extraction by itself with the rank rule on its spectrum (atp_principal_basis + atp_svd_entropy)
  attention    atp_attention on a basis the program already holds, with or without rotary positions
  linear       atp_lowrank_linear on a basis the program already holds
  alternating  atp_alternating_basis, the paper's Algorithm 1
  norm         atp_input_norm with a residual

listed() holds the benchmark's workloads and the small and odd calls beside them; draw() samples the same ranges.
Hidden states are a planted low-rank part plus noise, as in atp_inputs.py, made on the GPU from the seed.
"""
import math

import torch

import paper_2403_02352_b200 as atp
from paper_2403_02352_b200.layer import AtpLayer

DTYPES = {"f32": torch.float32, "bf16": torch.bfloat16}
POST_NORM = {"gelu": "layer", "swiglu": "rms", "": "layer"}


# ---------------------------------------------------------------------------------------------------- the cases
def listed():
    return [
        # prefill of one 4096-token prompt through a Llama-7B-like decoder layer at half the keys: the benchmark's
        # default size and the largest call
        {"name": "layer_llama_4096_r2048", "kind": "layer", "dtype": "bf16", "batch": 1, "L": 4096, "ragged": False,
         "div": 2, "r": 0, "heads": 32, "dh": 128, "d_ff": 11008, "ffn": "swiglu", "norm": "rms", "w_o": True,
         "spectrum": "geometric", "planted": 256, "noise": 0.01},
        # a batch of 16 short texts through a BERT-large-like encoder layer with its GELU FeedForward
        {"name": "layer_bert_large_b16_r256", "kind": "layer", "dtype": "bf16", "batch": 16, "L": 512, "ragged": False,
         "div": 2, "r": 0, "heads": 16, "dh": 64, "d_ff": 4096, "ffn": "gelu", "norm": "", "w_o": True,
         "spectrum": "geometric", "planted": 64, "noise": 0.02},
        # one text through a BERT-base-like attention block in fp32 at a quarter of the keys
        {"name": "layer_bert_base_f32_r128", "kind": "layer", "dtype": "f32", "batch": 1, "L": 512, "ragged": False,
         "div": 4, "r": 0, "heads": 12, "dh": 64, "d_ff": 0, "ffn": "", "norm": "", "w_o": True,
         "spectrum": "geometric", "planted": 32, "noise": 0.01},
        # serving: eight prompts of different lengths, extraction and attention with a quarter of each one's keys
        {"name": "serving_ragged_b8_1024", "kind": "layer", "dtype": "bf16", "batch": 8, "L": 1024, "ragged": True,
         "div": 4, "r": 0, "heads": 32, "dh": 128, "d_ff": 0, "ffn": "", "norm": "", "w_o": False,
         "spectrum": "geometric", "planted": 128, "noise": 0.01},
        # a long document with a fixed number of principal keys: extraction and attention only
        {"name": "long_context_32768_r1024", "kind": "layer", "dtype": "bf16", "batch": 1, "L": 32768, "ragged": False,
         "div": 0, "r": 1024, "heads": 32, "dh": 128, "d_ff": 0, "ffn": "", "norm": "", "w_o": False,
         "spectrum": "geometric", "planted": 512, "noise": 0.01},
        # choosing r for three texts of odd length: the leading spectrum and its entropy, with the basis itself
        {"name": "basis_odd_b3_701", "kind": "basis", "dtype": "bf16", "batch": 3, "L": 701, "ragged": True,
         "div": 0, "r": 96, "d": 1000, "spectrum": "geometric", "planted": 96, "noise": 0.01},
        # a second set of heads on a basis already extracted (4096 queries, 2048 keys)
        {"name": "attention_4096_r2048", "kind": "attention", "dtype": "bf16", "batch": 1, "L": 4096, "ragged": False,
         "div": 2, "r": 0, "heads": 32, "dh": 128, "rope": False, "full_q": False, "spectrum": "power", "planted": 256,
         "noise": 0.01},
        # rotary positions and exact queries over a ragged serving batch
        {"name": "attention_rope_ragged_b8", "kind": "attention", "dtype": "bf16", "batch": 8, "L": 1024, "ragged": True,
         "div": 4, "r": 0, "heads": 32, "dh": 128, "rope": True, "full_q": True, "spectrum": "geometric", "planted": 128,
         "noise": 0.01},
        # the gated FeedForward expansion of the Llama-7B-like layer
        {"name": "linear_swiglu_4096_r2048", "kind": "linear", "dtype": "bf16", "batch": 1, "L": 4096, "ragged": False,
         "div": 2, "r": 0, "d": 4096, "d_out": 11008, "act": "swiglu", "bias": False, "spectrum": "power",
         "planted": 256, "noise": 0.01},
        # the smallest call: one short text through one projection with bias and GELU, odd sizes
        {"name": "linear_short_77", "kind": "linear", "dtype": "bf16", "batch": 1, "L": 77, "ragged": False,
         "div": 4, "r": 0, "d": 768, "d_out": 3072, "act": "gelu", "bias": True, "spectrum": "geometric",
         "planted": 16, "noise": 0.02},
        # Algorithm 1 of the paper over a batch of short texts (two inner rounds, as the paper runs it)
        {"name": "alternating_b16_512_r64", "kind": "alternating", "dtype": "bf16", "batch": 16, "L": 512,
         "ragged": False, "div": 8, "r": 0, "d": 1024, "inner": 2, "spectrum": "geometric", "planted": 64,
         "noise": 0.02},
        # residual add and LayerNorm between attention and FeedForward of a long prompt
        {"name": "norm_residual_4096x4096", "kind": "norm", "dtype": "bf16", "rows": 4096, "d": 4096, "norm": "layer"},
    ]


def _log(rng, lo, hi):
    """An integer spread over the logarithm of its range."""
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["layer", "layer", "layer", "layer", "layer", "basis", "attention", "attention", "linear", "linear",
                       "alternating", "norm"])
    dtype = rng.choice(["bf16", "bf16", "bf16", "f32"])
    if kind == "norm":
        return {"kind": kind, "dtype": dtype, "rows": _log(rng, 16, 16384), "d": _log(rng, 256, 8192),
                "norm": rng.choice(["rms", "layer"])}
    # tokens of the call are bounded, and fp32 stays at encoder sizes (d up to 1024)
    small = dtype == "f32" or rng.random() < 0.5
    dh = 64 if small else 128
    heads = rng.choice([4, 8, 12, 16] if small else [8, 16, 32])
    L = _log(rng, 64, 1024 if small else 8192)
    batch = min(_log(rng, 1, 16), max(1, (8192 if small else 16384) // L))
    div = rng.choice([2, 4, 8])
    if not small and L > 4096:
        div = 8
    base = {"kind": kind, "dtype": dtype, "batch": batch, "L": L, "ragged": rng.random() < 0.5, "div": div, "r": 0,
            # a power law saturates the attention of long prompts: what is left of O after its leading directions, and
            # which of two tied keys a row takes, is then decided by rounding, whoever computes it
            "spectrum": rng.choice(["geometric", "power"]) if L <= 1024 else "geometric", "planted": _log(rng, 16, 256),
            "noise": rng.choice([0.01, 0.02])}
    d = heads * dh
    if kind == "layer":
        ffn = rng.choice(["", "gelu", "swiglu"]) if batch * L <= 4096 else ""
        base.update(heads=heads, dh=dh, ffn=ffn, d_ff=_log(rng, 2 * d, 4 * d) if ffn else 0,
                    norm=rng.choice(["", "rms"]), w_o=bool(ffn) or rng.random() < 0.5)
    elif kind == "basis":
        # the cut lies at the planted rank, where the components are determined by the input
        planted = min(_log(rng, 16, 128), L // 4)
        base.update(d=d + rng.choice([0, 8, 40]), div=0, r=planted, planted=planted, spectrum="geometric", noise=0.01)
    elif kind == "attention":
        base.update(heads=heads, dh=dh, rope=rng.random() < 0.3, full_q=rng.random() < 0.3)
    elif kind == "linear":
        act = rng.choice(["", "gelu", "swiglu"])
        base.update(d=d, d_out=_log(rng, d, 4 * d), act=act, bias=act != "swiglu" and rng.random() < 0.5)
    else:
        base.update(d=d, batch=min(batch, max(1, 8192 // L)), div=8, inner=rng.choice([1, 2, 3]))
        base["L"] = min(L, 1024)
    return base


# ---------------------------------------------------------------------------------------------------- sizes
def _lengths(case):
    L, n = case["L"], case["batch"]
    if not case["ragged"]:
        return [L] * n
    # spread over [L/2, L], the first sequence at full length
    return [L - int((b * 0.6180339887498949 % 1.0) * (L - L // 2)) for b in range(n)]


def _width(case):
    return case["heads"] * case["dh"] if "heads" in case else case["d"]


def _ranks(case):
    d = _width(case)
    return [max(1, min(case["r"] or L // case["div"], L, d, 2048)) for L in _lengths(case)]


# ---------------------------------------------------------------------------------------------------- inputs
def _padded(t):
    """Row-major copy whose leading dimension is a multiple of 8 elements, as the library asks for bf16."""
    rows, cols = t.shape
    out = torch.zeros((rows, (cols + 7) // 8 * 8), dtype=t.dtype, device=t.device)
    out[:, :cols] = t
    return out[:, :cols]


def _spectrum(case, k):
    i = torch.arange(k, dtype=torch.float32, device="cuda")
    if case["spectrum"] == "power":
        return (i + 1) ** -1.2
    return 10.0 ** (-2.0 * i / max(k - 1, 1))              # falls 100-fold over the planted part


def _orthonormal(gen, n, k):
    return torch.linalg.qr(torch.randn((n, k), generator=gen, device="cuda"))[0]


def _hidden(gen, case, L, d):
    """Planted low-rank part of unit mean square, plus noise."""
    k = min(case["planted"], L, d)
    s = _spectrum(case, k)
    s = s * math.sqrt(L * d) / torch.linalg.vector_norm(s)
    x = (_orthonormal(gen, L, k) * s) @ _orthonormal(gen, d, k).T
    return x + case["noise"] * torch.randn((L, d), generator=gen, device="cuda")


def _states(gen, case):
    return _padded(torch.cat([_hidden(gen, case, L, _width(case)) for L in _lengths(case)]).to(DTYPES[case["dtype"]]))


def _weight(gen, case, d_in, d_out):
    w = torch.randn((d_in, d_out), generator=gen, device="cuda").mul_(1 / math.sqrt(d_in))
    return _padded(w.to(DTYPES[case["dtype"]]))


def _kept_basis(gen, case):
    """A basis as an earlier extraction leaves it: orthonormal U_r, X_r = diag(sigma) V^T with the planted spectrum on
    top of the noise floor."""
    d, us, xs = _width(case), [], []
    width = (max(_ranks(case)) + 7) // 8 * 8
    for L, r in zip(_lengths(case), _ranks(case)):
        k = min(case["planted"], r)
        s = torch.zeros(r, device="cuda")
        s[:k] = _spectrum(case, k)
        s = s * math.sqrt(L * d) / torch.linalg.vector_norm(s)
        floor = case["noise"] * (math.sqrt(d) + math.sqrt(L)) * torch.linspace(1.0, 0.5, r, device="cuda")
        u = torch.zeros((L, width), device="cuda")
        u[:, :r] = _orthonormal(gen, L, r)
        us.append(u)
        xs.append(torch.sqrt(s * s + floor * floor)[:, None] * _orthonormal(gen, d, r).T)
    dt = DTYPES[case["dtype"]]
    return torch.cat(us).to(dt)[:, :max(_ranks(case))], _padded(torch.cat(xs).to(dt))


def prepare(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    ctx = atp.Context(0)
    st = {"case": case, "ctx": ctx}
    if case["kind"] == "norm":
        dt = DTYPES[case["dtype"]]
        st["X"] = _padded(torch.randn((case["rows"], case["d"]), generator=gen, device="cuda").to(dt))
        st["R"] = _padded(torch.randn((case["rows"], case["d"]), generator=gen, device="cuda").to(dt))
        st["out"] = _padded(torch.zeros_like(st["X"]))
        return st
    lengths, ranks, d = _lengths(case), _ranks(case), _width(case)
    st.update(lengths=lengths, ranks=ranks)
    if case["kind"] == "layer":
        names = {"W_Q": (d, d), "W_K": (d, d), "W_V": (d, d)}
        if case["w_o"]:
            names["W_O"] = (d, d)
        if case["ffn"] == "gelu":
            names.update(W_1=(d, case["d_ff"]), W_2=(case["d_ff"], d))
        elif case["ffn"] == "swiglu":
            names.update(W_gate=(d, case["d_ff"]), W_up=(d, case["d_ff"]), W_down=(case["d_ff"], d))
        weights = {n: _weight(gen, case, *shape) for n, shape in names.items()}
        st["layer"] = AtpLayer(ctx, weights, lengths, ranks, case["heads"], ffn=case["ffn"] or None,
                               input_norm=case["norm"] or None, post_norm=POST_NORM[case["ffn"]])
        st["X"] = _states(gen, case)
    elif case["kind"] == "attention":
        st["U"], st["Xr"] = _kept_basis(gen, case)
        st["X"] = _states(gen, case) if case["full_q"] else None
        st["W"] = [_weight(gen, case, d, d) for _ in range(3)]
        st["pos"] = torch.cat([torch.arange(L, dtype=torch.int32, device="cuda") for L in lengths]) if case["rope"] else None
    elif case["kind"] == "linear":
        st["U"], st["Xr"] = _kept_basis(gen, case)
        st["W"] = _weight(gen, case, d, case["d_out"])
        st["Wg"] = _weight(gen, case, d, case["d_out"]) if case["act"] == "swiglu" else None
        st["bias"] = torch.randn(case["d_out"], generator=gen, device="cuda") if case["bias"] else None
    elif case["kind"] == "alternating":
        st["X"] = _states(gen, case)
        st["V0"] = torch.randn((sum(ranks), d), generator=gen, device="cuda")
    else:
        st["X"] = _states(gen, case)
    return st


# ---------------------------------------------------------------------------------------------------- one pass
def run(st):
    case, ctx = st["case"], st["ctx"]
    kind = case["kind"]
    if kind == "layer":
        return st["layer"].forward(st["X"])
    if kind == "attention":
        return atp.atp_attention(ctx, st["X"], st["U"], st["Xr"], *st["W"], case["heads"], st["lengths"], st["ranks"],
                                 q_mode="full" if case["full_q"] else "lowrank",
                                 rope_base=10000.0 if case["rope"] else 0.0, positions=st["pos"])
    if kind == "linear":
        return atp.atp_lowrank_linear(ctx, st["U"], st["Xr"], st["W"], st["lengths"], st["ranks"], bias=st["bias"],
                                      act=case["act"] or None, W_gate=st["Wg"])
    if kind == "alternating":
        return atp.atp_alternating_basis(ctx, st["X"], st["V0"], st["lengths"], st["ranks"], inner=case["inner"])
    if kind == "norm":
        return atp.atp_input_norm(ctx, st["X"], st["R"], kind=case["norm"], out=st["out"])
    U, Xr, sigma = atp.atp_principal_basis(ctx, st["X"], st["lengths"], st["ranks"])
    mu, rank = atp.atp_svd_entropy(ctx, sigma, st["ranks"])
    return {"U": U, "X_r": Xr, "sigma": sigma, "mu": mu, "rank": rank}


# ---------------------------------------------------------------------------------------------------- work, tolerance
def work(case):
    """Floating-point operations of the method as it states them (an extraction: 4 L d r), every input read once and
    every output written once."""
    s = 2 if case["dtype"] == "bf16" else 4
    if case["kind"] == "norm":
        return {"bytes": 3 * case["rows"] * case["d"] * s, "flops": 8 * case["rows"] * case["d"]}
    d, flops, nbytes = _width(case), 0, 0
    kind = case["kind"]
    for L, r in zip(_lengths(case), _ranks(case)):
        if kind in ("layer", "basis"):
            flops += 4 * L * d * r
            nbytes += L * d * s
        if kind in ("layer", "attention"):
            flops += 6 * r * d * d + 2 * L * r * d + 4 * L * r * d
            nbytes += L * d * s
        if kind == "attention":
            nbytes += (L * r + r * d) * s
            if case["full_q"]:
                flops += 2 * L * d * d - 2 * L * r * d - 2 * r * d * d
                nbytes += L * d * s
            if case["rope"]:
                flops += 4 * L * r * d
        if kind == "layer":
            outs = [(d, d)] if case["w_o"] else []
            if case["ffn"]:
                outs += [(d, case["d_ff"] * (2 if case["ffn"] == "swiglu" else 1)), (case["d_ff"], d)]
            for d_in, d_out in outs:
                flops += 4 * L * d_in * r + 2 * r * d_in * d_out + 2 * L * r * d_out
        if kind == "linear":
            d_out = case["d_out"] * (2 if case["act"] == "swiglu" else 1)
            flops += 2 * r * d * d_out + 2 * L * r * d_out
            nbytes += (L * r + r * d + L * case["d_out"]) * s
        if kind == "alternating":
            flops += r * L * d * (4 * case["inner"] + 2)
            nbytes += (L * d + L * r + r * d) * s + r * d * 4
        if kind == "basis":
            nbytes += (L * r + r * d) * s
    if kind in ("layer", "attention"):
        nbytes += (4 if case.get("w_o") else 3) * d * d * s
    if kind == "layer" and case["ffn"]:
        nbytes += (3 if case["ffn"] == "swiglu" else 2) * d * case["d_ff"] * s
    if kind == "linear":
        nbytes += d * case["d_out"] * (2 if case["act"] == "swiglu" else 1) * s
    return {"bytes": nbytes, "flops": flops}


# Measured, then taken about fourfold. layer: against a run on the same rows in another order (every sum of the
# extraction in another order, the mathematics unchanged); bf16 layers with a FeedForward reach 2e-2 because each of the
# four extractions rounds its basis to bf16 and the next one starts from the result. basis: against the one-sided
# rotation (jacobi_block = 1). attention, linear, norm: against the same formulas in 64 bits. alternating: rows in
# another order agree to the last bit (64-bit sums), so the storage type's rounding is what another program may differ by.
TOLERANCE = {
    ("layer", "bf16"): {"rel": 3e-2, "max": 0.99},          # seen 2.1e-2, 0.7
    ("layer", "f32"): {"rel": 5e-4, "max": 2e-2},           # seen 1.4e-4, 3e-3
    ("basis", "bf16"): {"rel": 5e-3, "max": 6e-2},          # seen 1.4e-3, 1.4e-2
    ("basis", "f32"): {"rel": 2e-5, "max": 2e-4},           # seen 3.4e-6, 4.5e-5
    ("attention", "bf16"): {"rel": 1e-2, "max": 7e-2},      # seen 2.4e-3, 1.6e-2
    ("attention", "f32"): {"rel": 1e-5, "max": 2e-4},       # seen 1.4e-6, 4.3e-5
    ("linear", "bf16"): {"rel": 1.2e-2, "max": 0.3},        # seen 3.0e-3, 7.9e-2 (SwiGLU near the zero of the gate)
    ("linear", "f32"): {"rel": 5e-6, "max": 1e-4},          # seen 8.8e-7, 2.2e-5
    ("alternating", "bf16"): {"rel": 2e-3, "max": 2e-2},
    ("alternating", "f32"): {"rel": 1e-5, "max": 1e-3},
    ("norm", "bf16"): {"rel": 6e-3, "max": 1.6e-2},         # seen 1.7e-3, 3.9e-3
    ("norm", "f32"): {"rel": 5e-7, "max": 2e-6},            # seen 6e-8, 2.3e-7
}


def tolerance(case):
    return dict(TOLERANCE[case["kind"], case["dtype"]])
