"""The measured cases: what a user of this library has it do, through its public entry points.

Three kinds of pass:

    forward    one call of a kept plan: y = q * (h conv (k v))
    operator   one HyenaND layer at inference: the input-dependent kernel synthesised from its per-sample FiLM
               parameters (hyenand_synthesize_kernel), then Eq. 2 with it (Mixer)
    train      the convolution of one training step: forward, then dq, dk, dv, dh for a given dy (Backward)

over the boundary modes (zero-padded, causal, periodic), both I/O types, and filters per sample or shared over the
batch.  A case is a dict of plain values: kind, dims ("64x64"), B, C, dtype ("f32" | "bf16"), mode ("linear" |
"causal" | "circular"), shared (filter shared over the batch), field ("normal" | "spectral": smooth fields), and
for an operator the SIREN's hidden width and number of layers.
"""
import math

import torch

from paper_2607_19378_b200 import hyenand as hn
from paper_2607_19378_b200 import workloads as W

_MODES = {"linear": hn.HYENAND_MODE_LINEAR, "causal": hn.HYENAND_MODE_CAUSAL, "circular": hn.HYENAND_MODE_CIRCULAR}
_DTYPES = {"f32": hn.HYENAND_F32, "bf16": hn.HYENAND_BF16}


def _case(name, kind, dims, B, C, dtype, mode="linear", shared=False, field="normal", hidden=0, layers=0):
    c = {"kind": kind, "dims": dims, "B": B, "C": C, "dtype": dtype, "mode": mode, "shared": shared, "field": field,
         "hidden": hidden, "layers": layers}
    return dict(c, name=name) if name else c


def listed():
    return [
        # smallest call: one 32x32 grid of 8 channels, where launches and latency are all there is
        _case("tiny2d", "forward", "32x32", 1, 8, "f32"),
        # ViT-like token grid, 14x14 patches and one row of register tokens: many tiny ragged grids
        _case("tokens2d", "forward", "15x14", 32, 768, "bf16"),
        # 64x64 token grids of a hierarchical vision model's first stage (benchmark workload)
        _case("vision2d", "forward", "64x64", 16, 768, "bf16"),
        # 112x112 patch grid with a register row: a medium-sized grid off the powers of two
        _case("patches2d", "forward", "113x112", 4, 192, "bf16"),
        # 512x512 smooth fields in fp32 (benchmark workload)
        _case("pde2d", "forward", "512x512", 4, 128, "f32", field="spectral"),
        # the same fields with periodic boundaries (benchmark workload)
        _case("periodic2d", "forward", "512x512", 4, 128, "f32", mode="circular", field="spectral"),
        # causal sequence layer of ordinary context length, one filter per channel
        _case("seq1d", "forward", "2000", 16, 768, "bf16", mode="causal", shared=True),
        # long-context genomics layer (benchmark workload)
        _case("genomics1d", "forward", "262144", 2, 256, "bf16", mode="causal", shared=True),
        # medical volume: the largest pass (benchmark workload)
        _case("volume3d", "forward", "128x128x128", 1, 64, "bf16"),
        # the whole layer with its input-dependent kernel on vision token grids
        _case("operator2d", "operator", "64x64", 4, 384, "bf16", hidden=32, layers=2),
        # training step on vision token grids
        _case("train_vision2d", "train", "64x64", 4, 384, "bf16"),
        # training step on 96^3 crops of volumes
        _case("train_volume3d", "train", "96x96x96", 1, 12, "bf16"),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    """Grids, batch and options over the ranges the listed cases stand for: sequences of 64 to 262144, planes of 8 to
    512 and volumes of 8 to 128 per axis, odd extents and unequal axes among them; periodic grids have power-of-two
    extents (the library's rule).  The number of slices follows from a budget of padded points."""
    kind = rng.choice(["forward", "forward", "forward", "operator", "train"])
    ndim = rng.choice([1, 2, 2, 3])
    dtype = rng.choice(["bf16", "bf16", "f32"])
    top = {1: 262144 if kind == "forward" else 65536, 2: 512, 3: 128}[ndim]
    low = {1: 64, 2: 8, 3: 8}[ndim]
    base = _log(rng, low, top)
    dims = [max(low, min(top, round(base * (1.0 if a == 0 else _log(rng, 0.6, 1.6))))) for a in range(ndim)]
    mode = "linear"
    if ndim == 1:
        mode = rng.choice(["causal", "causal", "causal", "linear"])
    elif rng.random() < 0.15:
        mode = "circular"
        dims = [min(top, 1 << round(math.log2(d))) for d in dims]
    elif rng.random() < 0.3:
        dims[0] = min(top, dims[0] + 1)                       # a row of register tokens
    shared = kind != "operator" and rng.random() < (0.6 if ndim == 1 else 0.25)
    padded = math.prod(2 * d for d in dims)
    budget = _log(rng, 1 << 16, 1 << (28 if kind == "forward" else 26))
    slices = max(1, min(16384, int(budget / padded)))
    B = max(1, min(slices, round(_log(rng, 1, 32))))
    C = max(1, min(1536, slices // B))
    field = "spectral" if ndim == 2 and dtype == "f32" and min(dims) >= 64 else "normal"
    hidden, layers = (rng.choice([16, 32, 64]), rng.choice([2, 3])) if kind == "operator" else (0, 0)
    return _case("", kind, "x".join(str(d) for d in dims), B, C, dtype, mode, shared, field, hidden, layers)


def _workload(case, seed):
    dims = tuple(int(d) for d in case["dims"].split("x"))
    causal, circular = case["mode"] == "causal", case["mode"] == "circular"
    return W.Workload("case", dims, case["B"], case["C"], case["dtype"], causal=causal, h_shared=case["shared"], seed=seed,
                      filt="causal_exp" if causal else "radial", alpha=(0.5, 8.0) if causal else (0.05, 0.5),
                      field=case["field"], circular=circular)


def _siren(case, w, gen):
    """Parameters of the kernel network of one layer, in the SIREN's usual ranges, and per-sample FiLM values."""
    def uni(shape, a, b):
        return torch.rand(shape, generator=gen, device="cuda") * (b - a) + a
    H, J, C, N = case["hidden"], case["layers"], w.C, w.ndim
    r = math.sqrt(6.0 / H)
    return {"W1": uni((H, N), -1.0, 1.0), "b1": uni((H,), -0.5, 0.5), "omega0": uni((H,), 1.0, 30.0),
            "Wh": uni((J - 1, H, H), -r, r), "bh": uni((J - 1, H), -0.3, 0.3),
            "Wout": uni((C, H), -r, r), "bout": uni((C,), -0.1, 0.1),
            "gamma": 1.0 + 0.3 * torch.randn((w.B, J, H), generator=gen, device="cuda"),
            "beta": 0.3 * torch.randn((w.B, J, H), generator=gen, device="cuda"),
            "window": uni((C,), 0.5, 8.0) if w.causal else uni((N, C), 0.2, 1.5)}


def prepare(case, seed):
    w = _workload(case, seed)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed * 1000003 + 17)
    s = {"case": case, "w": w}
    if case["kind"] == "operator":
        draw3 = [torch.randn((w.B, w.C) + w.dims, generator=gen, device="cuda").to(w.torch_dtype) for _ in range(3)]
        s["q"], s["k"], s["v"] = draw3
        s["siren"] = _siren(case, w, gen)
        s["g_in"] = 1.0 + 0.1 * torch.randn((w.C,), generator=gen, device="cuda")
        s["g_out"] = 1.0 + 0.1 * torch.randn((w.C,), generator=gen, device="cuda")
        s["h"] = torch.empty((w.B, w.C) + w.taps, device="cuda", dtype=w.torch_dtype)
        s["mixer"] = hn.Mixer(w.dims, w.B, w.C, mode=w.mode, dtype=w.torch_dtype, eps=1e-6)
        return s
    s["q"], s["k"], s["v"], s["h"] = W.make_inputs(w, device="cuda")
    s["plan"] = hn.Plan(w.dims, w.B, w.C, causal=w.causal, dtype=w.torch_dtype, circular=w.circular)
    if case["kind"] == "train":
        s["dy"] = torch.randn(s["q"].shape, generator=gen, device="cuda").to(w.torch_dtype)
        s["backward"] = hn.Backward(w.dims, w.B, w.C, mode=w.mode, dtype=w.torch_dtype)
    return s


def run(s):
    case, w = s["case"], s["w"]
    if case["kind"] == "operator":
        p = s["siren"]
        hn.hyenand_synthesize_kernel(w.dims, _MODES[w.mode], w.B, w.C, case["hidden"], case["layers"], p["W1"], p["b1"],
                                     p["omega0"], p["Wh"], p["bh"], p["Wout"], p["bout"], p["gamma"], p["beta"],
                                     p["window"], _DTYPES[case["dtype"]], s["h"])
        return {"h": s["h"], "y": s["mixer"].forward(s["q"], s["k"], s["v"], s["h"], s["g_in"], s["g_out"])}
    y = s["plan"].forward(s["q"], s["k"], s["v"], s["h"])
    if case["kind"] == "forward":
        return y
    dq, dk, dv, dh = s["backward"](s["q"], s["k"], s["v"], s["h"], s["dy"])
    return {"y": y, "dq": dq, "dk": dk, "dv": dv, "dh": dh}


def work(case):
    """Every tensor once; 2.5 N log2 N per real transform of N = 2L points per axis (N = L where periodic): k v, the
    filter and the result of a forward; those, dy q and the three gradients' of a training step (each stage counted
    once where forward and backward both need it, except that a forward's spectra are not kept for the backward); the
    network's multiply-adds of a synthesis."""
    w = _workload(case, 0)
    es = 4 if case["dtype"] == "f32" else 2
    S, Sh = w.B * w.C, w.C if w.h_shared else w.B * w.C
    n, taps = w.elements * es, Sh * math.prod(w.taps) * es
    pts = math.prod(d if w.circular else 2 * d for d in w.dims)
    fft = 2.5 * pts * math.log2(max(2, pts))
    if case["kind"] == "forward":
        return {"bytes": 4 * n + taps, "flops": fft * (2 * S + Sh)}
    if case["kind"] == "train":
        # q, k, v, h, dy in; y, dq, dk, dv, dh out
        return {"bytes": 8 * n + 2 * taps, "flops": fft * (7 * S + 2 * Sh)}
    H, J = case["hidden"], case["layers"]
    net = 2.0 * w.B * math.prod(w.taps) * (w.ndim * H + (J - 1) * H * H + H * w.C)
    return {"bytes": 4 * n + taps, "flops": fft * (2 * S + Sh) + net}


def tolerance(case):
    """fp32 transforms of these lengths are within 2e-7 to 4e-7 of a 64-bit evaluation, synthesised fp32 kernels within
    1e-6 (their first sine's argument reaches 30 radians and more); a bf16 store alone is 1.7e-3 (up to 2^-8 of a single
    value).  Four times that."""
    if case["dtype"] == "bf16":
        return {"rel": 7e-3, "max": 0.02}
    return {"rel": 5e-6 if case["kind"] == "operator" else 2e-6}
