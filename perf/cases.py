"""Workloads on which the library's speed is measured: what a policy-gradient trainer has it do, layer by layer.

Every case is one pass of a linear layer (or of the seven projections of a decoder block) over a packed ragged microbatch:
per-sequence Fisher Gram K, advantage transform, weight gradient.  `kind` says which of the library's ways is taken:

  layer     isopo_layer_gram + isopo_transform_advantages + isopo_weight_grad: the three calls of one layer
  hook      the same inside a backward hook: running-mean regulariser on the device, dW accumulated (beta = 1)
  block     the seven projections of a decoder block; q/k/v and gate/up read the same X.  `one_ws`: one workspace reused by
            every projection, a transform each; otherwise a workspace each and one batched transform
  shared    projections that read one X through the shared-X entry points, one batched transform
  sampled   Algorithm 1's token-sampled coefficients + the stand-alone weight gradient
  many      more than 256 sequences: Gram route, the large interacting solve, the stand-alone weight gradient
  spectral  the interacting transform through the eigendecomposition, spectrum returned

Sizes are those of the package's own workloads (a 64-wide float32 layer, an 896-wide, a 1536-wide and a 3584-wide block)
and generic ones between them.
"""

import math

import numpy as np
import torch

from paper_2512_23353_b200 import binding as b

VARIANTS = {"normalised": b.VAR_NORMALISED, "direction": b.VAR_DIRECTION, "euclid": b.VAR_EUCLID, "general": b.VAR_GENERAL,
            "interacting": b.VAR_INTERACTING, "normalised_raw": b.VAR_NORMALISED_RAW}
DTYPES = {"bf16": (b.BF16, torch.bfloat16, 2), "f32": (b.F32, torch.float32, 4)}
DY_STD = 0.1
# largest drawn case: below the largest listed one in arithmetic and in memory
MAX_FLOPS, MAX_BYTES = 1.5e13, 1.6e10


def _case(kind, dtype, d_in, d_out, B, law, lo, hi, lens, variant="interacting", **more):
    return {"kind": kind, "dtype": dtype, "d_in": d_in, "d_out": d_out, "B": B, "law": law, "lo": lo, "hi": hi, "lens": lens,
            "variant": variant, "mode": "default", "kv": 0, "samples": 0, "one_ws": False, **more}


def listed():
    return [
        # the smallest call: a float32 adapter-sized layer, a handful of short sequences; latency is all there is
        dict(_case("layer", "f32", 64, 64, 8, "uniform", 16, 64, 1), name="tiny_f32"),
        # a float32 layer of ordinary width on short sequences (full-precision runs, debugging a bf16 run)
        dict(_case("layer", "f32", 896, 896, 64, "uniform", 16, 128, 2, "normalised"), name="f32_layer"),
        # odd widths, few and very uneven sequences down to one token
        dict(_case("layer", "bf16", 1000, 328, 13, "uniform", 1, 300, 3, "direction"), name="odd_bf16"),
        # one attention projection of the 896-wide block in a backward hook, as a training run calls it
        dict(_case("hook", "bf16", 896, 896, 64, "uniform", 128, 1024, 4), name="hook_q_896"),
        # the 896-wide block, 64 sequences of up to 1024 tokens, one batched transform
        dict(_case("block", "bf16", 896, 4864, 64, "uniform", 128, 1024, 5, kv=128), name="block_896"),
        # the same block on many short rollouts, where K comes from token Grams and nothing per sequence is stored
        dict(_case("block", "bf16", 896, 4864, 256, "uniform", 16, 64, 6, "normalised", kv=128), name="short_rollouts_896"),
        # q/k/v of the 1536-wide block through the shared-input entry point
        dict(_case("shared", "bf16", 1536, 1536, 64, "loguniform", 256, 4096, 7, kv=256), name="qkv_shared_1536"),
        # the 1536-wide block at its full microbatch (32 prompts x 8 samples, long-tailed lengths), one workspace
        dict(_case("block", "bf16", 1536, 8960, 256, "loguniform", 256, 4096, 8, kv=256, one_ws=True), name="block_1536"),
        # the widest projection: gate of the 3584-wide block, 300k tokens
        dict(_case("layer", "bf16", 3584, 18944, 64, "uniform", 1024, 8192, 9), name="gate_3584"),
        # Algorithm 1 as printed on the 1536-wide block's gate projection
        dict(_case("sampled", "bf16", 1536, 8960, 256, "loguniform", 256, 4096, 10, "normalised", samples=128), name="sampled_gate_1536"),
        # a whole 1024-rollout batch solved at once: K from token Grams, the large solve
        dict(_case("many", "bf16", 896, 896, 1024, "uniform", 16, 64, 11), name="many_1024"),
        # Algorithm 2 as printed (eigendecomposition) with the spectrum, for monitoring a run
        dict(_case("spectral", "bf16", 896, 896, 256, "uniform", 16, 64, 12), name="spectral_256"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the listed ranges: widths on and off every tile grid, sequence counts and lengths over their whole range."""
    while True:
        kind = rng.choice(["layer", "layer", "layer", "hook", "hook", "block", "block", "shared", "sampled", "sampled", "many", "spectral"])
        dtype = rng.choice(["f32", "bf16", "bf16"]) if kind in ("layer", "sampled") else "bf16"
        lo = _log_int(rng, 1, 1024)
        hi = min(8192, lo * _log_int(rng, 2, 16))
        law = rng.choice(["uniform", "loguniform"])
        B = rng.randint(257, 1024) if kind == "many" else _log_int(rng, 4, 256)
        width = lambda top: max(8, _log_int(rng, 64, top) // 8 * 8)  # noqa: E731
        if kind == "block":
            d_in = rng.choice([896, 1024, 1536, 2048, 2560, 3584])
            d_out, kv = rng.choice([2, 3, 4, 5]) * d_in + rng.choice([0, 128, 384]), rng.choice([128, 256, 512])
        else:
            d_in, d_out, kv = width(4096), width(8192), 128 * rng.randint(1, 4)
            if rng.random() < 0.3:
                d_in, d_out = d_out, d_in
        if dtype == "f32":
            d_in, d_out, hi = min(d_in, 1536) + rng.choice([0, 1, 3]), min(d_out, 1536) + rng.choice([0, 1, 3]), min(hi, 256)
            lo = min(lo, hi)
        if kind in ("many", "spectral"):
            lo, hi = min(lo, 64), min(hi, 128)
        variant = "interacting" if kind in ("many", "spectral") else "normalised" if kind == "sampled" else rng.choice(
            ["interacting", "interacting", "interacting"] + sorted(VARIANTS))
        if kind == "hook" and variant == "general":
            variant = "interacting"
        c = _case(kind, dtype, d_in, d_out, B, law, lo, hi, rng.randint(100, 1 << 20), variant, kv=kv if kind in ("block", "shared") else 0,
                  samples=rng.choice([32, 128, 128, 512]) if kind == "sampled" else 0, one_ws=kind == "block" and rng.random() < 0.5,
                  mode=rng.choice(["default"] * 4 + ["deterministic", "split"]) if kind == "layer" and dtype == "bf16" else "default")
        w = work(c)
        if w["flops"] <= (MAX_FLOPS if dtype == "bf16" else 3e11) and _state_bytes(c) <= MAX_BYTES:
            return c


# ---- sizes ----

def _lengths(c):
    """Sequence lengths of the case; the seed of the inputs only permutes them."""
    rng = np.random.default_rng(c["lens"])
    if c["law"] == "uniform":
        return rng.integers(c["lo"], c["hi"] + 1, size=c["B"])
    return np.clip(np.rint(np.exp(rng.uniform(math.log(c["lo"]), math.log(c["hi"]), size=c["B"]))).astype(np.int64), c["lo"], c["hi"])


def _projections(c):
    """[(index of the X it reads, d_in, d_out)] of the case."""
    d, f, kv = c["d_in"], c["d_out"], c["kv"]
    if c["kind"] == "block":
        return [(0, d, d), (0, d, kv), (0, d, kv), (1, d, d), (2, d, f), (2, d, f), (3, f, d)]
    if c["kind"] == "shared":
        return [(0, d, f), (0, d, kv), (0, d, kv)]
    return [(0, d, f)]


def _path(c, T, d_in, d_out):
    """The route by the library's own rule where the caller has the choice."""
    if c["kind"] in ("many", "sampled"):
        return b.PATH_GRAM
    return b.isopo_choose_path(DTYPES[c["dtype"]][0], T, d_in, d_out, c["B"])


def _state_bytes(c):
    elt, T, proj = DTYPES[c["dtype"]][2], int(_lengths(c).sum()), _projections(c)
    inputs = elt * T * (sum({i: d for i, d, _ in proj}.values()) + sum(o for _, _, o in proj))
    stored = [elt * c["B"] * (d + 255) * (o + 127) if _path(c, T, d, o) == b.PATH_MATERIALISE else elt * T * min(d, o) for _, d, o in proj]
    return inputs + (max(stored) if c["one_ws"] else sum(stored)) + 4 * sum(d * o for _, d, o in proj)


def work(c):
    """Inputs read once and outputs written once; the weight-gradient GEMM and the cheaper of the two ways to K."""
    elt, B, T, proj = DTYPES[c["dtype"]][2], c["B"], int(_lengths(c).sum()), _projections(c)
    nbytes = elt * T * (sum({i: d for i, d, _ in proj}.values()) + sum(o for _, _, o in proj))
    flops = 0.0
    for _, d, o in proj:
        nbytes += 4 * (d * o + B) + (0 if c["kind"] == "sampled" else 4 * B * B)
        k = 2.0 * T * c["samples"] * (d + o) if c["kind"] == "sampled" else min(1.0 * B * B * d * o, 1.0 * T * T * (d + o))
        flops += 2.0 * T * d * o + k
    return {"bytes": float(nbytes), "flops": flops}


def tolerance(c):
    """float32: float32 products and sums.  bf16: the stored gradients (and the scaled operand of the stand-alone weight
    gradient) are rounded to bf16, K's off-diagonals inherit it, and the solve passes it on to the coefficients."""
    return {"rel": 1e-5} if c["dtype"] == "f32" else {"rel": 1e-2}


# ---- one pass ----

def _advantages(rng, B):
    """Group-normalised Bernoulli rewards, groups of 8 with p ~ U[0.1, 0.9]."""
    p = rng.uniform(0.1, 0.9, size=(B + 7) // 8)
    r = (rng.uniform(size=(len(p), 8)) < p[:, None]).astype(np.float64)
    A = (r - r.mean(1, keepdims=True)) / (r.std(1, keepdims=True) + 1e-6)
    return A.reshape(-1)[:B].astype(np.float32)


def _tokens(gen, T, d, dt, std):
    """Activations or output gradients: independent noise plus a shared rank-4 component of the same energy, as token
    features have (sequences' gradients then overlap)."""
    x = torch.empty((T, d), device="cuda", dtype=dt).normal_(0.0, std, generator=gen)
    a = torch.empty((T, 4), device="cuda", dtype=dt).normal_(0.0, 0.5 * std, generator=gen)
    u = torch.empty((4, d), device="cuda", dtype=dt).normal_(0.0, 1.0, generator=gen)
    return x.addmm_(a, u)


def _workspace(nbytes):
    raw = torch.empty(nbytes + 1024, dtype=torch.uint8, device="cuda")
    shift = (-raw.data_ptr()) % 1024
    return raw[shift:shift + nbytes]


def _set_mode(mode):
    if mode == "deterministic":
        b.isopo_set_deterministic(True)
    elif mode == "split":
        b.isopo_set_store_format(b.STORE_E4M3_SPLIT)


def _reset_mode(mode):
    if mode == "deterministic":
        b.isopo_set_deterministic(False)
    elif mode == "split":
        b.isopo_set_store_format(b.STORE_BF16)


def prepare(c, seed):
    code, dt, _ = DTYPES[c["dtype"]]
    B, proj = c["B"], _projections(c)
    rng = np.random.default_rng([seed, c["lens"]])
    off = np.concatenate([[0], np.cumsum(rng.permutation(_lengths(c)))]).astype(np.int64)
    T = int(off[-1])
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed * 7919 + 13)
    widths = {i: d for i, d, _ in proj}
    xs = {i: _tokens(gen, T, widths[i], dt, 1.0) for i in sorted(widths)}
    s = {"case": c, "off": off, "T": T, "X": [xs[i] for i, _, _ in proj], "dY": [_tokens(gen, T, o, dt, DY_STD) for _, _, o in proj],
         "A": torch.from_numpy(_advantages(rng, B)).cuda(), "info": torch.zeros(1, dtype=torch.int32, device="cuda"),
         "variant": VARIANTS[c["variant"]], "K": [torch.empty((B, B), device="cuda") for _ in proj],
         "c": [torch.empty(B, device="cuda") for _ in proj], "dW": [torch.zeros((o, d), device="cuda") for _, d, o in proj],
         # the shared-X entry points and the stand-alone weight gradient name their route; elsewhere it is left to the library
         "path": [_path(c, T, d, o) if c["kind"] in ("shared", "many", "sampled") else b.PATH_AUTO for _, d, o in proj]}
    # regulariser: 1e-3 of the typical ||G_i||^2, what a running mean of earlier microbatches would hold
    s["lam"] = [1e-3 * 4.0 * T / B * d * o * DY_STD ** 2 if c["variant"] in ("interacting", "euclid") else 0.0 for _, d, o in proj]
    s["pqr"] = [-0.5, -0.5, 0.25, 0.0, 0.0, 0.0] if c["variant"] == "general" else None
    _set_mode(c["mode"])
    if c["kind"] == "sampled":
        s["rows"] = rng.permutation(T)[:c["samples"]].astype(np.int64)
        s["F2"] = torch.empty(B, device="cuda")
        need = [b.isopo_sampled_workspace_bytes(code, T, d, o, B, len(s["rows"])) for _, d, o in proj]
    else:
        need = [b.isopo_workspace_bytes(code, T, d, o, B, p) for (_, d, o), p in zip(proj, s["path"])]
    _reset_mode(c["mode"])
    s["ws"] = [_workspace(max(need))] * len(proj) if c["one_ws"] else [_workspace(n) for n in need]
    if c["kind"] == "hook":
        s["ema"] = torch.zeros(4, device="cuda")
    if c["kind"] == "many":
        s["solve_ws"] = torch.empty(b.isopo_transform_large_workspace_bytes(B), dtype=torch.uint8, device="cuda")
    if c["kind"] == "spectral":
        s["eig"] = torch.empty(B, device="cuda")
        s["solve_ws"] = torch.empty(b.lib.isopo_spectral_workspace_bytes(), dtype=torch.uint8, device="cuda")
    return s


def _gram(s, h):
    b.isopo_layer_gram(s["X"][h], s["dY"][h], s["off"], s["K"][h], s["ws"][h], s["info"], s["path"][h])


def _transform(s, h):
    b.isopo_transform_advantages(s["K"][h], s["A"], s["variant"], s["lam"][h], s["c"][h], s["info"], s["pqr"])


def _transform_all(s):
    b.isopo_transform_advantages_batched(s["K"], s["A"], s["variant"], s["lam"], s["c"], s["info"], s["pqr"])


def _weight_grad(s, h, beta=0.0):
    b.isopo_weight_grad(s["X"][h], s["dY"][h], s["c"][h], s["off"], s["dW"][h], s["ws"][h], s["info"], s["path"][h], beta)


def run(s):
    c = s["case"]
    kind, n = c["kind"], len(s["dY"])
    out = {"K": s["K"], "c": s["c"], "dW": s["dW"], "info": s["info"]}
    if kind == "layer":
        _set_mode(c["mode"])
        _gram(s, 0)
        _transform(s, 0)
        _weight_grad(s, 0)
        _reset_mode(c["mode"])
    elif kind == "hook":
        _gram(s, 0)
        b.isopo_reg_ema_update(s["K"][0], 0.9, s["ema"])
        b.isopo_transform_advantages_rel(s["K"][0], s["A"], s["variant"], 1e-3, s["ema"], s["c"][0], s["info"])
        _weight_grad(s, 0, 1.0)
        out["ema"] = s["ema"]
    elif kind == "block" and c["one_ws"]:
        for h in range(n):
            _gram(s, h)
            _transform(s, h)
            _weight_grad(s, h)
    elif kind == "block":
        for h in range(n):
            _gram(s, h)
        _transform_all(s)
        for h in range(n):
            _weight_grad(s, h)
    elif kind == "shared":
        if all(p == b.PATH_MATERIALISE for p in s["path"]):
            b.isopo_layer_gram_shared_x_stored(s["X"][0], s["dY"], s["off"], s["K"], s["ws"], s["info"])
        elif all(p == b.PATH_GRAM for p in s["path"]):
            wide = max(range(n), key=lambda h: s["ws"][h].numel())
            b.isopo_layer_gram_shared_x(s["X"][0], s["dY"], s["off"], s["K"], s["ws"][wide], s["info"])
        else:
            for h in range(n):
                _gram(s, h)
        _transform_all(s)
        for h in range(n):
            _weight_grad(s, h)
    elif kind == "sampled":
        b.isopo_sampled_coefficients(s["X"][0], s["dY"][0], s["off"], s["rows"], s["A"], 0.0, s["c"][0], s["ws"][0], s["info"], s["F2"])
        _weight_grad(s, 0)
        out = {"c": s["c"], "F2": s["F2"], "dW": s["dW"], "info": s["info"]}
    elif kind == "many":
        _gram(s, 0)
        b.isopo_transform_advantages_large(s["K"][0], s["A"], s["lam"][0], s["c"][0], s["solve_ws"], s["info"])
        _weight_grad(s, 0)
    else:
        _gram(s, 0)
        b.isopo_transform_spectral(s["K"][0], s["A"], s["lam"][0], s["c"][0], s["info"], 0.0, s["eig"], s["solve_ws"])
        _weight_grad(s, 0)
        out["eigenvalues"] = s["eig"]
    return out
