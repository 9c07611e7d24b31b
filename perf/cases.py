"""The work this library is measured on: what a program that quantizes or runs a model's
linear layers has it do, through the public entry points (`pipeline.LayerPipeline` and the
calls of `kronq`). Sizes are those of the repository's own layer configurations, tests and
benchmark, or generic ones; inputs follow the repository's synthetic recipe (lognormal
channel scales with outlier channels, Gaussian weights with rare large entries), drawn on
the GPU from the seed.

Kinds of case:
  layer    one whole layer, `LayerPipeline.run`: factors, rescale, rotations, inverse
           Cholesky, sweep
  factor   the online statistic H = A^T A of one input, its tokens arriving in chunks
  rotate   the two-sided incoherence rotations of a layer's weights and of its H_X
  chol     the damped inverse Cholesky factor of H_X
  sweep    the column-wise quantization of rotated weights with L, either trailing update,
           per-row or group grids, with or without the drift correction
  drift    the drift statistic, its rotation and the correction matrix P
  decode   one decode step of a quantized transformer block's seven linear sublayers, as a
           captured CUDA graph (what a serving loop replays)
  infer    one quantized layer applied to a batch of tokens by a direct call
"""
import math

import numpy as np
import torch

from paper_2607_07964_gb300 import kronq as kq
from paper_2607_07964_gb300.pipeline import LayerPipeline

DEV = "cuda"
DAMP = 0.01
ALPHA = 0.25
OUTLIERS = 16


def listed():
    return [
        # the smallest whole layer (the repository's oracle-size layer): launches and latency
        {"name": "layer_256", "kind": "layer", "d_out": 256, "d_in": 256, "tokens": 4096, "bits": 4, "group": 0},
        # an 8B attention projection over 64 calibration sequences of 2048 tokens: an ordinary layer
        {"name": "layer_4096", "kind": "layer", "d_out": 4096, "d_in": 4096, "tokens": 131072, "bits": 4,
         "group": 128},
        # the output-gradient factor of a 70B k/v projection: few features, many tokens
        {"name": "factor_1024", "kind": "factor", "d": 1024, "tokens": 262144, "chunk": 262144},
        # a wide MLP input whose calibration tokens arrive in two chunks, the last one ragged
        {"name": "factor_14336", "kind": "factor", "d": 14336, "tokens": 12000, "chunk": 8192},
        # the rotations of an 8B down projection (rows of 28 * 512)
        {"name": "rotate_14336", "kind": "rotate", "d_out": 4096, "d_in": 14336},
        # the inverse Cholesky of an 8B down projection's H_X: the largest one here
        {"name": "chol_14336", "kind": "chol", "n": 14336},
        # the sweep of a 70B k/v projection: few rows, long rows, 2-bit group grids
        {"name": "sweep_1024x8192", "kind": "sweep", "d_out": 1024, "d_in": 8192, "bits": 2, "group": 128,
         "trailing": "3xtf32", "drift": False},
        # the sweep of an 8B gate/up projection: many rows, 3-bit group grids
        {"name": "sweep_14336x4096", "kind": "sweep", "d_out": 14336, "d_in": 4096, "bits": 3, "group": 128,
         "trailing": "3xtf32", "drift": False},
        # the bit-exact fp32 sweep on sizes that fit no tile, per-row grids
        {"name": "sweep_ragged_fp32", "kind": "sweep", "d_out": 1000, "d_in": 2001, "bits": 4, "group": 0,
         "trailing": "fp32", "drift": False},
        # the drift correction of an 8B attention projection
        {"name": "drift_4096", "kind": "drift", "d": 4096, "tokens": 32768},
        # one token through the seven linear sublayers of an 8B block at 4 bits
        {"name": "decode_8b_4bit", "kind": "decode", "d_model": 4096, "d_kv": 1024, "d_ff": 14336, "bits": 4,
         "batch": 1},
        # eight tokens through an 8B down projection at 2 bits
        {"name": "infer_8_tokens", "kind": "infer", "d_out": 4096, "d_in": 14336, "bits": 2, "group": 128, "batch": 8},
    ]


# Lengths with a Hadamard construction, 2^k and 28 * 2^k.
HADAMARD = [256, 448, 512, 896, 1024, 1792, 2048, 3584, 4096, 7168, 8192, 14336]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["layer", "factor", "rotate", "chol", "sweep", "drift", "decode", "infer"])
    if kind == "layer":
        d_out, d_in = (rng.choice([h for h in HADAMARD if h <= 8192]) for _ in range(2))
        top = min(131072, int(4.0e12 / (d_out * d_out + d_in * d_in)))
        return {"kind": kind, "d_out": d_out, "d_in": d_in, "tokens": _log(rng, 2000, top), "bits": rng.choice([2, 3, 4]),
                "group": rng.choice([0, 128])}
    if kind == "factor":
        d = _log(rng, 200, 14336)
        tokens = _log(rng, 1000, min(262144, int(4.0e12 / (d * d))))
        return {"kind": kind, "d": d, "tokens": tokens, "chunk": rng.choice([tokens, max(512, tokens // 3)])}
    if kind == "rotate":
        return {"kind": kind, "d_out": rng.choice(HADAMARD), "d_in": rng.choice(HADAMARD)}
    if kind == "chol":
        return {"kind": kind, "n": _log(rng, 200, 14336)}
    if kind == "sweep":
        drift = rng.random() < 0.25
        trailing = rng.choice(["3xtf32", "3xtf32", "fp32"])
        d_in = _log(rng, 200, 8192)
        step = 16 if drift else 4 if trailing == "3xtf32" else 1
        d_in = max(step, d_in // step * step)
        d_out = _log(rng, 100, min(14336, int(6.0e10 / (d_in * d_in)) + 100) if trailing == "fp32" else
                     min(14336, 50_000_000 // d_in))
        return {"kind": kind, "d_out": d_out, "d_in": d_in, "bits": rng.choice([2, 3, 4, 8]), "group": rng.choice([0, 128]),
                "trailing": trailing, "drift": drift}
    if kind == "drift":
        d = rng.choice([h for h in HADAMARD if h <= 8192])
        return {"kind": kind, "d": d, "tokens": _log(rng, 1000, min(65536, int(1.0e12 / (d * d))))}
    if kind == "decode":
        m = rng.choice([256, 512, 1024, 1792, 2048, 3584, 4096])
        ff = rng.choice([h for h in HADAMARD if 2 * m <= h <= 4 * m])
        return {"kind": kind, "d_model": m, "d_kv": rng.choice([m, m // 4]), "d_ff": ff, "bits": rng.choice([2, 3, 4, 8]),
                "batch": rng.choice([1, 1, 2, 4])}
    hads = [h for h in HADAMARD if h % 128 == 0]
    return {"kind": kind, "d_out": rng.choice(HADAMARD), "d_in": rng.choice(hads), "bits": rng.choice([2, 3, 4, 8]),
            "group": rng.choice([0, 128]), "batch": rng.randint(1, 8)}


# ------------------------------------------------------------------------------- inputs
class _Draw:
    """Seeded inputs on the GPU."""

    def __init__(self, seed):
        self.g = torch.Generator(device=DEV)
        self.g.manual_seed(int(seed) * 7919 + 17)

    def normal(self, *shape):
        return torch.randn(shape, generator=self.g, device=DEV)

    def uniform(self, *shape):
        return torch.rand(shape, generator=self.g, device=DEV)

    def scales(self, d, sigma, outliers=0):
        s = torch.exp(sigma * self.normal(d))
        if outliers:
            s[torch.randperm(d, generator=self.g, device=DEV)[:outliers]] *= 20.0
        return s

    def tokens(self, T, d, scale):
        """[T, d] bf16 in rows padded to a multiple of 8 elements (what the factor calls ask for)."""
        ld = (d + 7) // 8 * 8
        out = torch.zeros((T, ld), dtype=torch.bfloat16, device=DEV)[:, :d]
        step = max(1, (1 << 26) // d)
        for t in range(0, T, step):
            n = min(step, T - t)
            out[t:t + n] = (self.normal(n, d) * scale).to(torch.bfloat16)
        return out

    def weights(self, d_out, d_in):
        w = 0.02 * self.normal(d_out, d_in)
        return torch.where(self.uniform(d_out, d_in) < 0.001, w * 10.0, w)

    def signs(self, d):
        return ((self.uniform(d) < 0.5).to(torch.int8) * 2 - 1).contiguous()

    def second_moment(self, n):
        """H = X^T X over 2 n tokens of correlated channels (a rotated H_X: even diagonal)."""
        r = max(1, n // 8)
        mix = self.normal(r, n)
        x = self.normal(2 * n, n) + self.normal(2 * n, r) @ mix / math.sqrt(r) * 2.0
        h = x.T @ x
        return (h + h.T) * 0.5


def _damped(h, damp):
    h = h.double()
    h.diagonal().add_(damp * h.diagonal().mean())
    return h


def _inverse_factor(h64):
    """Lower L with h64^-1 = L L^T: the Cholesky factor of the index-reversed matrix, inverted."""
    n = h64.shape[0]
    c = torch.linalg.cholesky(h64.flip(0, 1))
    z = torch.linalg.solve_triangular(c, torch.eye(n, dtype=torch.float64, device=h64.device), upper=False)
    del c
    return z.T.flip(0, 1)


def _quantized(d, d_out, d_in, bits, group):
    """A quantized layer as the sweep leaves it: packed codes, grids, scales and signs."""
    ng = 1 if group == 0 else d_in // group
    top = 2 ** bits - 1
    q = torch.clamp(torch.round(d.normal(d_out, d_in) * (top / 6.0) + top / 2.0), 0, top).to(torch.uint8)
    packed = torch.empty(kq.kq_packed_codes_bytes(d_out, d_in, bits) // 4, dtype=torch.int32, device=DEV)
    kq.kq_pack_codes(q, bits, packed)
    return {"codes": q, "packed": packed, "scale": 0.12 / top * (0.5 + d.uniform(d_out, ng)),
            "zero": torch.round(top / 2.0 + (d.uniform(d_out, ng) - 0.5) * top / 4.0).to(torch.int32),
            "s_x": torch.exp(0.5 * d.normal(d_in)), "s_g": torch.exp(0.5 * d.normal(d_out)),
            "su": d.signs(d_out), "sv": d.signs(d_in), "d_out": d_out, "d_in": d_in, "bits": bits, "group": group}


def _empty(*shape, dtype=torch.float32):
    return torch.empty(shape, dtype=dtype, device=DEV)


def _ws(n):
    return torch.empty((max(1, n),), dtype=torch.uint8, device=DEV)


# The sublayers of a block: (name, whose output it reads or "x", d_out, d_in).
def _sublayers(case):
    m, kv, ff = case["d_model"], case["d_kv"], case["d_ff"]
    return [("q", "x", m, m), ("k", "x", kv, m), ("v", "x", kv, m), ("o", "q", m, m), ("gate", "o", ff, m),
            ("up", "o", ff, m), ("down", "up", m, ff)]


def _inputs(case, seed):
    """The inputs of a case, without the library's buffers (exact() uses the same)."""
    d, k = _Draw(seed), case["kind"]
    if k == "layer":
        o, i, T = case["d_out"], case["d_in"], case["tokens"]
        return {"X": d.tokens(T, i, d.scales(i, 1.0, OUTLIERS)), "G": d.tokens(T, o, d.scales(o, 1.5)), "W": d.weights(o, i),
                "su": d.signs(o), "sv": d.signs(i)}
    if k == "factor":
        return {"A": d.tokens(case["tokens"], case["d"], d.scales(case["d"], 1.0, OUTLIERS))}
    if k == "rotate":
        o, i = case["d_out"], case["d_in"]
        x = d.normal(256, i) * d.scales(i, 1.0, OUTLIERS)
        return {"W": d.weights(o, i), "H": x.T @ x, "s_x": d.scales(i, 0.5), "s_g": d.scales(o, 0.5),
                "su": d.signs(o), "sv": d.signs(i)}
    if k == "chol":
        return {"H": d.second_moment(case["n"])}
    if k == "sweep":
        o, i = case["d_out"], case["d_in"]
        s = {"W": d.normal(o, i) * 0.02, "Lt": _inverse_factor(_damped(d.second_moment(i), DAMP)).float().contiguous(),
             "Pt": None}
        if case["drift"]:
            s["Pt"] = torch.tril(d.normal(i, i) * (0.05 / math.sqrt(i)), -1).contiguous()
        return s
    if k == "drift":
        n, T = case["d"], case["tokens"]
        scale = d.scales(n, 1.0, OUTLIERS)
        X = d.tokens(T, n, scale)
        Xt = torch.empty_like(X)
        step = max(1, (1 << 26) // n)
        for t in range(0, T, step):
            m = min(step, T - t)
            Xt[t:t + m] = (X[t:t + m].float() + 0.1 * scale * d.normal(m, n)).to(torch.bfloat16)
        return {"X": X, "Xt": Xt, "s_x": torch.sqrt(scale), "sv": d.signs(n),
                "Lt": _inverse_factor(_damped(d.second_moment(n), DAMP)).float().contiguous()}
    if k == "decode":
        return {"x": d.normal(case["batch"], case["d_model"]),
                "layers": {name: _quantized(d, o, i, case["bits"], 128) for name, _, o, i in _sublayers(case)}}
    return {"x": d.normal(case["batch"], case["d_in"]),
            "layer": _quantized(d, case["d_out"], case["d_in"], case["bits"], case["group"])}


def _infer(L, x, y, ws, stream=None):
    kq.kq_infer(L["packed"], L["scale"], L["zero"], L["d_out"], L["d_in"], L["bits"], L["group"], L["s_x"], L["s_g"],
                L["su"], L["sv"], x, y, ws, stream=stream)


def prepare(case, seed):
    s, k = _inputs(case, seed), case["kind"]
    s["kind"] = k
    if k == "layer":
        s["pipe"] = LayerPipeline(case["d_out"], case["d_in"], case["bits"], case["group"], device=DEV)
    elif k == "factor":
        s["chunk"] = case["chunk"]
        s["H"], s["trace"], s["info"] = _empty(case["d"], case["d"]), _empty(1, dtype=torch.float64), _zero_word()
    elif k == "rotate":
        s["Wp"], s["Hp"] = torch.empty_like(s["W"]), torch.empty_like(s["H"])
    elif k == "chol":
        s["Lt"], s["info"], s["ws"] = torch.empty_like(s["H"]), _zero_word(), _ws(kq.kq_chol_inv_workspace(case["n"]))
    elif k == "sweep":
        o, i, g = case["d_out"], case["d_in"], case["group"]
        ng = 1 if g == 0 else -(-i // g)
        s["mode"] = kq.KQ_TRAIL_FP32 if case["trailing"] == "fp32" else kq.KQ_TRAIL_3XTF32
        s["bits"], s["group"], s["Wp"] = case["bits"], g, torch.empty_like(s["W"])
        s["codes"], s["scale"] = _empty(o, i, dtype=torch.uint8), _empty(o, ng)
        s["zero"], s["col_loss"], s["info"] = _empty(o, ng, dtype=torch.int32), _empty(i), _zero_word()
        s["ws"] = _ws(kq.kq_obs_quantize_workspace(o, i, 128, s["mode"], case["drift"]))
    elif k == "drift":
        n = case["d"]
        s["D"], s["Pt"], s["info"] = _empty(n, n), _empty(n, n), _zero_word()
        s["ws_d"], s["ws_p"] = _ws(kq.kq_accum_drift_workspace(case["tokens"], n)), _ws(kq.kq_gptaq_p_workspace(n))
    elif k == "decode":
        b = case["batch"]
        s["y"] = {name: _empty(b, o) for name, _, o, _ in _sublayers(case)}
        s["wss"] = {name: _ws(kq.kq_infer_workspace(b, i, o)) for name, _, o, i in _sublayers(case)}

        def step(stream):
            for name, src, _, _ in _sublayers(case):
                _infer(s["layers"][name], s["x"] if src == "x" else s["y"][src], s["y"][name], s["wss"][name], stream)

        step(torch.cuda.current_stream())
        torch.cuda.synchronize()
        s["graph"], cap = torch.cuda.CUDAGraph(), torch.cuda.Stream()
        with torch.cuda.graph(s["graph"], stream=cap):
            step(cap)
    else:
        s["y"] = _empty(case["batch"], case["d_out"])
        s["ws"] = _ws(kq.kq_infer_workspace(case["batch"], case["d_in"], case["d_out"]))
    return s


def _zero_word():
    return torch.zeros(1, dtype=torch.int32, device=DEV)


def run(s):
    k = s["kind"]
    if k == "layer":
        p = s["pipe"]
        p.run(s["X"], s["G"], s["W"], s["su"], s["sv"])
        return {"codes": p.codes, "scale": p.scale, "zero": p.zero, "col_loss": p.col_loss, "s_x": p.s_x, "s_g": p.s_g,
                "traces": p.traces}
    if k == "factor":
        T = s["A"].shape[0]
        for t in range(0, T, s["chunk"]):
            e = min(T, t + s["chunk"])
            kq.kq_accum_factor(s["A"][t:e], s["H"], accumulate=t > 0, trace=s["trace"] if e == T else None, info=s["info"])
        return {"H": s["H"], "trace": s["trace"]}
    if k == "rotate":   # the raw factor and weights stay as they are, as in LayerPipeline.run_from_factors
        s["Hp"].copy_(s["H"])
        s["Wp"].copy_(s["W"])
        kq.kq_rotate_in(s["Wp"], s["Hp"], s["s_x"], s["sv"], kq.KQ_FWD_SYM)
        kq.kq_rotate_out(s["Wp"], None, s["s_g"], s["su"], kq.KQ_FWD)
        return {"W": s["Wp"], "H": s["Hp"]}
    if k == "chol":
        kq.kq_chol_inv(s["H"], DAMP, s["Lt"], s["info"], s["ws"])
        return {"Lt": s["Lt"]}
    if k == "sweep":   # the sweep destroys W'
        s["Wp"].copy_(s["W"])
        kq.kq_obs_quantize(s["Wp"], s["Lt"], s["bits"], s["group"], 128, s["codes"], s["scale"], s["zero"], s["col_loss"],
                           None, s["ws"], mode=s["mode"], info=s["info"], Pt=s["Pt"])
        return {"codes": s["codes"], "scale": s["scale"], "zero": s["zero"], "col_loss": s["col_loss"]}
    if k == "drift":
        kq.kq_accum_drift(s["Xt"], s["X"], s["D"], info=s["info"], ws=s["ws_d"])
        kq.kq_rotate_in(None, s["D"], s["s_x"], s["sv"], kq.KQ_FWD)
        kq.kq_gptaq_p(s["D"], s["Lt"], ALPHA, s["Pt"], s["ws_p"], info=s["info"])
        return {"D": s["D"], "Pt": s["Pt"]}
    if k == "decode":
        s["graph"].replay()
        return s["y"]
    _infer(s["layer"], s["x"], s["y"], s["ws"])
    return s["y"]


# --------------------------------------------------------------------------------- work
def _grid_bytes(d_out, d_in, group):
    return 8 * d_out * (1 if group == 0 else -(-d_in // group))


def _layer_bytes(d_out, d_in, bits, group, batch):
    return (d_out * d_in * (4 if bits == 3 else bits) / 8 + _grid_bytes(d_out, d_in, group) + 5 * (d_out + d_in) +
            4 * batch * (d_out + d_in))


def work(case):
    k = case["kind"]
    if k == "layer":
        o, i, T = case["d_out"], case["d_in"], case["tokens"]
        return {"bytes": 2 * T * (o + i) + 5 * o * i + _grid_bytes(o, i, case["group"]) + 9 * i + 5 * o,
                "flops": T * (i * (i + 1) + o * (o + 1)) + 2 * i ** 3 / 3 + o * i * max(0, i - 128) +
                2 * o * i * math.log2(o * i) + 4 * i * i * math.log2(i)}
    if k == "factor":
        d, T = case["d"], case["tokens"]
        return {"bytes": 2 * T * d + 4 * d * d, "flops": T * d * (d + 1)}
    if k == "rotate":
        o, i = case["d_out"], case["d_in"]
        return {"bytes": 8 * (o * i + i * i) + 5 * (o + i), "flops": o * i * math.log2(o * i) + 2 * i * i * math.log2(i)}
    if k == "chol":   # the lower triangle in, the whole L out
        n = case["n"]
        return {"bytes": 6 * n * n, "flops": 2 * n ** 3 / 3}
    if k == "sweep":
        o, i = case["d_out"], case["d_in"]
        m = 2 if case["drift"] else 1
        return {"bytes": 5 * o * i + m * 2 * i * i + _grid_bytes(o, i, case["group"]) + 4 * i, "flops": m * o * i * i}
    if k == "drift":
        n, T = case["d"], case["tokens"]
        return {"bytes": 4 * T * n + 10 * n * n, "flops": 2 * T * n * n + 2 * n ** 3 / 3 + 2 * n * n * math.log2(n)}
    b = case["batch"]
    shapes = [(o, i, 128) for _, _, o, i in _sublayers(case)] if k == "decode" else [(case["d_out"], case["d_in"], case["group"])]
    return {"bytes": sum(_layer_bytes(o, i, case["bits"], g, b) for o, i, g in shapes),
            "flops": sum(2 * b * o * i + b * (o * math.log2(o) + i * math.log2(i)) for o, i, _ in shapes)}


# ------------------------------------------------------------------------------ 64 bits
def _paley28():
    """The Hadamard matrix of order 28 of Paley's second construction over GF(13)."""
    squares = {x * x % 13 for x in range(1, 13)}
    q = np.array([[0 if i == j else (1 if (j - i) % 13 in squares else -1) for j in range(13)] for i in range(13)])
    c = np.ones((14, 14), dtype=np.int64)
    c[0, 0], c[1:, 1:] = 0, q
    return np.kron(c, [[1, 1], [1, -1]]) + np.kron(np.eye(14, dtype=np.int64), [[1, -1], [-1, -1]])


def _hadamard(v):
    """H_n applied to the last axis (Sylvester for 2^k, H_28 (x) H_2^k for 28 * 2^k) over sqrt(n)."""
    n = v.shape[-1]
    a = 28 if n % 28 == 0 else 1
    p = n // a
    lead = v.shape[:-1]
    x, h = v.reshape(-1, a, p), 1
    while h < p:
        x = x.reshape(-1, a, p // (2 * h), 2, h)
        x = torch.stack((x[..., 0, :] + x[..., 1, :], x[..., 0, :] - x[..., 1, :]), dim=-2)
        h *= 2
    x = x.reshape(-1, a, p)
    if a == 28:
        x = torch.matmul(torch.from_numpy(_paley28()).double().to(v.device), x)
    return x.reshape(*lead, n) / math.sqrt(n)


def _two_sided(m, s, sign):
    """V S^-1 M S^-1 V^T."""
    f = sign.double() / s.double()
    m = _hadamard(m * f).T
    return _hadamard(m * f).T


def _cross64(a, b):
    out = torch.zeros((a.shape[1], b.shape[1]), dtype=torch.float64, device=a.device)
    step = max(1, (1 << 27) // a.shape[1])
    for t in range(0, a.shape[0], step):
        out.addmm_(a[t:t + step].double().T, b[t:t + step].double())
    return out


def _infer64(L, x):
    o, i = L["d_out"], L["d_in"]
    g = i if L["group"] == 0 else L["group"]
    xr = _hadamard(x.double() / L["s_x"].double() * L["sv"].double())
    y = torch.empty((x.shape[0], o), dtype=torch.float64, device=x.device)
    step = max(1, (1 << 26) // i)
    for r in range(0, o, step):
        q = L["codes"][r:r + step].double().reshape(-1, i // g, g)
        q = (q - L["zero"][r:r + step].double()[..., None]) * L["scale"][r:r + step].double()[..., None]
        y[:, r:r + step] = xr @ q.reshape(-1, i).T
    return _hadamard(y) * L["su"].double() / L["s_g"].double()


def exact(case, seed):
    k = case["kind"]
    if k == "sweep":   # its outputs are decisions, each on those before it
        return None
    s = _inputs(case, seed)
    if k == "layer":   # the scales and traces; the codes and grids are decisions
        def diag(a):
            out, step = torch.zeros(a.shape[1], dtype=torch.float64, device=DEV), max(1, (1 << 26) // a.shape[1])
            for t in range(0, a.shape[0], step):
                out += a[t:t + step].double().square().sum(0)
            return out

        hx, hg, w2 = diag(s["X"]), diag(s["G"]), s["W"].double().square()
        s_x, s_g = (hx / w2.sum(0)) ** 0.25, (hg / w2.sum(1)) ** 0.25
        t = [hx.sum(), hg.sum(), hx.sum() * hg.sum(), (hx / s_x ** 2).sum(), (hg / s_g ** 2).sum()]
        return {"codes": None, "scale": None, "zero": None, "col_loss": None, "s_x": s_x, "s_g": s_g,
                "traces": torch.stack(t + [t[3] * t[4]])}
    if k == "factor":
        h = _cross64(s["A"], s["A"])
        return {"H": h, "trace": h.diagonal().sum().reshape(1)}
    if k == "rotate":
        w = _hadamard(s["W"].double() * s["s_x"].double() * s["sv"].double())
        w = _hadamard((w * s["s_g"].double()[:, None] * s["su"].double()[:, None]).T).T
        return {"W": w, "H": _two_sided(s["H"].double(), s["s_x"], s["sv"])}
    if k == "chol":
        return {"Lt": _inverse_factor(_damped(s["H"], DAMP))}
    if k == "drift":
        dx = (s["Xt"].float() - s["X"].float())
        d = _two_sided(_cross64(dx, s["X"]), s["s_x"], s["sv"])
        L = s["Lt"].double()
        return {"D": d, "Pt": (ALPHA * torch.triu(d @ L, 1) @ L.T).T}
    if k == "decode":
        y = {}
        for name, src, _, _ in _sublayers(case):
            y[name] = _infer64(s["layers"][name], s["x"] if src == "x" else y[src])
        return y
    return _infer64(s["layer"], s["x"])
