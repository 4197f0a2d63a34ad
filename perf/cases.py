"""The measured work of the BaKron library: what a quantisation run has it do, layer by layer.

A layer goes through three steps, each one public call: its Hessian factors are
accumulated from calibration samples (``kfac_factors``, ``shampoo_factors``,
``bakron_gram``), factored once (``bakron_prepare``) and its weights rounded
(``bakron_solve`` and its forms).  The sizes are those of the workloads and tests
here: 128 x 128 up to 4096 x 11008, ragged sides among them.

``listed`` gives the fixed cases, ``draw`` more of the same ranges, ``prepare`` what a
program holds before the call, ``run`` one pass, ``work`` its unavoidable bytes and
flops, ``exact`` its outputs in 64 bits.

The factors behind a solve are made here with torch and handed over by
``bakron_set_factors``, as a program does that keeps them on disk, so that a solve is
measured on the same factors whatever ``bakron_prepare`` does.
"""
import math

import torch

import paper_2608_06291_gb300 as P

DTYPES = {"f32": torch.float32, "bf16": torch.bfloat16}


def listed():
    return [
        # Hessian factors of a 4096-wide projection from eight sequences of 2048 tokens
        {"name": "kfac_16k_tokens", "path": "kfac", "k": 16384, "m": 4096, "n": 4096, "x": "bf16"},
        # one sequence's samples added to the running Gram of an MLP input
        {"name": "gram_add_11008", "path": "gram", "k": 2048, "n": 11008, "x": "bf16", "beta": 1.0},
        # the weighted factors, fp32 samples, no side a multiple of a tile
        {"name": "shampoo_ragged", "path": "shampoo", "k": 5000, "m": 1000, "n": 1531, "x": "f32"},
        # the factorisation of a 4096-wide projection's Grams, and of a small ragged layer's
        {"name": "prepare_4096", "path": "prepare", "m": 4096, "n": 4096, "damp": 0.01},
        {"name": "prepare_ragged", "path": "prepare", "m": 1000, "n": 1531, "damp": 0.5},
        # the smallest call: one 128 x 128 layer, everything at its default
        {"name": "solve_128", "path": "solve", "m": 128, "n": 128, "w": "f32", "bits": 4, "group": 0,
         "pre": True, "keep": False},
        # a small layer with sides of no tile's multiple, 3 bits, the rounded-at values kept
        {"name": "solve_ragged", "path": "solve", "m": 1000, "n": 1531, "w": "f32", "bits": 3, "group": 0,
         "pre": True, "keep": False},
        # an attention projection, and an MLP down-projection with groups of 128: the
        # layers most of a model's time goes to, workspace kept from layer to layer
        {"name": "solve_4096", "path": "solve", "m": 4096, "n": 4096, "w": "bf16", "bits": 4, "group": 0,
         "pre": False, "keep": True},
        {"name": "solve_mlp_down_g128", "path": "solve", "m": 4096, "n": 11008, "w": "bf16", "bits": 4,
         "group": 128, "pre": False, "keep": True},
        # the symmetric alphabet with shrunk scales, then the solve on that grid
        {"name": "symmetric_2048x4096", "path": "symmetric", "m": 2048, "n": 4096, "w": "bf16", "levels": 3},
        # GPTQ (no output-side factor) of an attention projection
        {"name": "gptq_4096_g128", "path": "gptq", "m": 4096, "n": 4096, "w": "bf16", "bits": 4, "group": 128},
        # the heads of one attention layer side by side, each with its own output-side factor
        {"name": "heads_32x128x4096", "path": "heads", "h": 32, "m": 128, "n": 4096, "w": "bf16", "bits": 4},
    ]


def _size(rng, lo, hi):
    """A side of lo .. hi, spread over its logarithm; a third of them multiples of 128."""
    v = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    if rng.random() < 0.34 and v >= 128:
        v = v // 128 * 128
    return max(lo, min(hi, v))


def draw(rng):
    path = rng.choice(["kfac", "gram", "shampoo", "prepare", "solve", "solve", "solve", "symmetric",
                       "gptq", "gptq", "heads"])
    if path == "kfac":
        return {"path": path, "k": _size(rng, 256, 16384), "m": _size(rng, 64, 4096), "n": _size(rng, 64, 4096),
                "x": rng.choice(["bf16", "bf16", "f32"])}
    if path == "gram":
        return {"path": path, "k": _size(rng, 256, 8192), "n": _size(rng, 64, 8192), "x": rng.choice(["bf16", "f32"]),
                "beta": rng.choice([0.0, 1.0])}
    if path == "shampoo":
        return {"path": path, "k": _size(rng, 256, 8192), "m": _size(rng, 64, 4096), "n": _size(rng, 64, 4096),
                "x": rng.choice(["bf16", "f32"])}
    if path == "prepare":
        return {"path": path, "m": _size(rng, 64, 4096), "n": _size(rng, 64, 4096), "damp": rng.choice([0.01, 0.5])}
    if path == "heads":
        return {"path": path, "h": rng.randint(2, 32), "m": rng.choice([64, 128]), "n": _size(rng, 256, 4096),
                "w": rng.choice(["bf16", "f32"]), "bits": rng.choice([2, 3, 4])}
    m, n = _size(rng, 64, 4096), _size(rng, 64, 8192)
    w = rng.choice(["bf16", "f32"])
    if path == "symmetric":
        return {"path": path, "m": m, "n": min(n, 4096), "w": w, "levels": rng.choice([1, 3, 7])}
    group = rng.choice([0, 0, 32, 64, 128])
    if group:
        n = max(group, n // group * group)
    c = {"path": path, "m": m, "n": n, "w": w, "bits": rng.choice([2, 3, 4, 8]), "group": group}
    if path == "solve":
        c["pre"] = rng.random() < 0.3
        c["keep"] = rng.random() < 0.5
    return c


# ------------------------------------------------------------------ inputs
def _gen(seed, part):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) * 16 + part)
    return g


def _samples(k, d, alpha, g):
    """k samples of d features (fp32) with a power-law spectrum: a few strong directions, each
    spread over every feature, over a floor of independent noise."""
    r = min(d, 512)
    lam = torch.arange(1, r + 1, device="cuda", dtype=torch.float32).pow(-alpha / 2)
    mix = torch.randn(r, d, generator=g, device="cuda") / math.sqrt(r)
    z = torch.randn(k, r, generator=g, device="cuda")
    return (z * lam) @ mix + 0.05 * torch.randn(k, d, generator=g, device="cuda")


def _gram(d, alpha, g):
    x = _samples(2048, d, alpha, g)
    return x.T @ x / x.shape[0]


def _factor(d, alpha, g, damp=0.01):
    """The unit-lower factor (fp32) of a damped Gram: H = R^T R, R lower, and R^-1 diag(R)."""
    h = _gram(d, alpha, g).double()
    h.diagonal().add_(damp * h.diagonal().mean())
    r = torch.linalg.cholesky(h.flip(0, 1)).flip(0, 1).T.float()     # lower, R^T R = H
    eye = torch.diag(r.diagonal())
    return torch.linalg.solve_triangular(r, eye, upper=False).tril()


def _weights(m, n, dtype, g):
    """Weights of a linear layer: Gaussian, one column in a thousand ten times as large."""
    w = 0.02 * torch.randn(m, n, generator=g, device="cuda")
    cols = torch.randperm(n, generator=g, device="cuda")[: max(1, n // 1000)]
    w[:, cols] *= 10.0
    return w.to(DTYPES[dtype])


def prepare(case, seed):
    path = case["path"]
    s = {"case": case}
    if path in ("kfac", "shampoo"):
        s["a"] = _samples(case["k"], case["n"], 1.0, _gen(seed, 0)).to(DTYPES[case["x"]])
        s["b"] = _samples(case["k"], case["m"], 0.5, _gen(seed, 1)).to(DTYPES[case["x"]])
    elif path == "gram":
        s["x"] = _samples(case["k"], case["n"], 1.0, _gen(seed, 0)).to(DTYPES[case["x"]])
        s["g"] = _gram(case["n"], 1.0, _gen(seed, 1)) if case["beta"] else None
    elif path == "prepare":
        s["A"] = _gram(case["n"], 1.0, _gen(seed, 0))
        s["B"] = _gram(case["m"], 0.5, _gen(seed, 1))
    elif path == "heads":
        m, n, h = case["m"], case["n"], case["h"]
        la = _factor(n, 1.0, _gen(seed, 0))
        w = _weights(h * m, n, case["w"], _gen(seed, 1))
        s["W"] = [w[i * m:(i + 1) * m] for i in range(h)]
        g = _gen(seed, 2)
        s["f"] = [P.bakron_set_factors(la, _factor(m, 0.5, g)) for _ in range(h)]
        s["ws"] = torch.empty(P.bakron_batched_workspace_bytes(m, n, h), dtype=torch.uint8, device="cuda")
    else:
        m, n = case["m"], case["n"]
        la = _factor(n, 1.0, _gen(seed, 0))
        lb = torch.eye(m, device="cuda") if path == "gptq" else _factor(m, 0.5, _gen(seed, 1))
        s["W"] = _weights(m, n, case["w"], _gen(seed, 2))
        s["f"] = P.bakron_set_factors(la, lb)
        if path != "solve" or case["keep"]:
            s["ws"] = P.alloc_workspace(m, n)
        if path == "solve" and case["pre"] and m * n <= 20000:
            s["L"] = (la, lb)
    return s


# -------------------------------------------------------------------- one pass
def run(state):
    c = state["case"]
    path = c["path"]
    if path == "kfac":
        return P.kfac_factors(state["a"], state["b"])
    if path == "shampoo":
        return P.shampoo_factors(state["a"], state["b"])
    if path == "gram":
        return P.bakron_gram(state["x"], alpha=1.0 / c["k"], beta=c["beta"], G=state["g"], sync=False)
    if path == "prepare":
        f = P.bakron_prepare(state["A"], state["B"], c["damp"])
        return P.bakron_get_factors(f)
    if path == "solve":
        if c["keep"]:
            return P.bakron_solve(state["W"], state["f"], c["bits"], c["group"], workspace=state["ws"],
                                  prerounding=c["pre"], sync=False)
        return P.bakron_solve(state["W"], state["f"], c["bits"], c["group"], prerounding=c["pre"])
    if path == "symmetric":
        scales, zeros = P.bakron_grid_symmetric(state["W"], c["levels"])
        codes = P.bakron_solve_with_grid(state["W"], state["f"], scales, zeros, 2 * c["levels"],
                                         workspace=state["ws"], sync=False)
        return codes, scales, zeros
    if path == "gptq":
        return P.bakron_solve_gptq(state["W"], state["f"], c["bits"], c["group"], workspace=state["ws"],
                                   sync=False)
    h, m, n = c["h"], c["m"], c["n"]
    codes = torch.empty(h, m, n, dtype=torch.uint8, device="cuda")
    grid = torch.empty(2, h, m, 1, dtype=torch.float32, device="cuda")
    P.bakron_solve_batched(state["W"], state["f"], c["bits"], streams=h, workspace=state["ws"],
                           out=list(zip(codes, grid[0], grid[1])), sync=False)
    return codes, grid[0], grid[1]


# ------------------------------------------------------------------------ work
def work(case):
    """Each input read and each output written once (of a symmetric or triangular matrix that is
    read: one half), and the multiply-adds of the definition: a Gram's distinct entries; a Cholesky
    and a triangular inverse; per rounded entry the errors above it and left of it."""
    path = case["path"]
    xb = 4 if case.get("x", case.get("w")) == "f32" else 2
    n, m = case["n"], case.get("m", 0)
    if path in ("kfac", "shampoo"):
        k = case["k"]
        return {"bytes": xb * k * (n + m) + 4 * (n * n + m * m), "flops": float(k) * (n * (n + 1) + m * (m + 1))}
    if path == "gram":
        k = case["k"]
        return {"bytes": xb * k * n + 4 * n * n * (1.5 if case["beta"] else 1.0), "flops": float(k) * n * (n + 1)}
    if path == "prepare":
        return {"bytes": 6 * (n * n + m * m), "flops": 2.0 / 3.0 * (float(n) ** 3 + float(m) ** 3)}
    h = case.get("h", 1)
    per = (xb + 1 + (4 if case.get("pre") else 0)) * m * n
    if path == "gptq":
        return {"bytes": per + 2 * n * n, "flops": float(m) * n * (n - 1)}
    return {"bytes": h * (per + 2 * m * m) + 2 * n * n, "flops": float(h) * m * n * (m + n)}


# --------------------------------------------------------------- in 64 bits
def _grid64(w, bits, group):
    m, n = w.shape
    v = w.double().reshape(m, -1, group or n)
    lo, hi = v.amin(2).clamp(max=0), v.amax(2).clamp(min=0)
    flat = (lo == 0) & (hi == 0)
    lo, hi = torch.where(flat, -torch.ones_like(lo), lo), torch.where(flat, torch.ones_like(hi), hi)
    s = (hi - lo) / (2 ** bits - 1)
    return s, torch.round(-lo / s)


def _rounded_at64(w, la, lb, s, z, qmax):
    """Codes and pre-rounding values, one anti-diagonal after the other; `inb` holds what the
    entries rounded so far send to each."""
    m, n = w.shape
    s, z = (t.repeat_interleave(n // t.shape[1], 1) for t in (s, z))
    w, la, lb = w.double(), la.double(), lb.double()
    inb, x, codes = torch.zeros_like(w), torch.zeros_like(w), torch.zeros(m, n, dtype=torch.uint8, device=w.device)
    for k in range(m + n - 1):
        i = torch.arange(max(0, k - n + 1), min(m, k + 1), device=w.device)
        j = k - i
        at = w[i, j] + inb[i, j]
        c = (torch.round(at / s[i, j]) + z[i, j]).clamp(0, qmax)
        e = s[i, j] * (c - z[i, j]) - at
        x[i, j], codes[i, j] = at, c.to(torch.uint8)
        inb += (lb[:, i] * e) @ la[:, j].T
    return codes, x


def _symmetric64(w, levels, steps=50):
    """Among the scales amax (2K - k) / (2K l), each rounded as a float of 32 bits is, the one of
    the least squared error."""
    amax = w.float().abs().amax(1)
    amax = torch.where(amax == 0, torch.ones_like(amax), amax)
    v = w.double()
    best, err = None, None
    for k in range(steps + 1):
        t = torch.tensor((2 * steps - k) / (2 * steps * levels), dtype=torch.float32, device=w.device)
        s = (amax * t).double()[:, None]
        d = ((torch.round(v / s).clamp(-levels, levels) * s - v) ** 2).sum(1)
        best = s[:, 0] if best is None else torch.where(d < err, s[:, 0], best)
        err = d if err is None else torch.minimum(d, err)
    return best[:, None], torch.full_like(best, float(levels))[:, None]


def _prepare64(h, damp):
    h = h.double().tril()
    h = h + h.tril(-1).T
    h.diagonal().add_(damp * h.diagonal().mean())
    r = torch.linalg.cholesky(h.flip(0, 1)).flip(0, 1).T
    d = r.diagonal().clone()
    return torch.linalg.solve_triangular(r, torch.diag(d), upper=False).tril(), d


def exact(case, seed):
    path = case["path"]
    s = prepare(case, seed)
    if path in ("kfac", "shampoo"):
        a, b = s["a"].double(), s["b"].double()
        wa, wb = (((b * b).sum(1), (a * a).sum(1)) if path == "shampoo" else (1.0, 1.0))
        one = lambda x, w: (x.T if isinstance(w, float) else x.T * w) @ x / case["k"]  # noqa: E731
        return one(a, wa), one(b, wb)
    if path == "gram":
        x = s["x"].double()
        g = x.T @ x / case["k"]
        return g + s["g"].double() if case["beta"] else g
    if path == "prepare":
        la, ra = _prepare64(s["A"], case["damp"])
        lb, rb = _prepare64(s["B"], case["damp"])
        return la, lb, ra, rb
    if path == "symmetric":
        scales, zeros = _symmetric64(s["W"], case["levels"])
        return None, scales, zeros
    # one flipped near-tie sends every later entry another way, so the rounded values themselves
    # have a 64-bit answer only where no tie is likely: in the small problems
    if path == "heads":
        scales, zeros = _grid64(torch.cat(s["W"]), case["bits"], 0)
        return None, scales.reshape(case["h"], -1, 1), zeros.reshape(case["h"], -1, 1)
    scales, zeros = _grid64(s["W"], case["bits"], case["group"])
    if path == "solve" and case["pre"]:
        if "L" not in s:
            return None, scales, zeros, None
        codes, x = _rounded_at64(s["W"], *s["L"], scales, zeros, 2 ** case["bits"] - 1)
        return codes, scales, zeros, x
    return None, scales, zeros
