"""The work this framework is measured on: calls of its public entry points,
on inputs made on the GPU from a seed.

A case is a dict with ``call`` (the entry point), the matrix family and its
sizes, and the series with its options.  The families and sizes are those of
the repository's workloads, benchmark and tests: 1D Laplacians, 2D five-point
operators on rectangular grids (up to 512 x 512), symmetric banded random
matrices, the banded N(0, 1) family, unstructured sparse matrices whose powers
fill in, batches of small instances, and a burst of serving requests.
"""
import math
import random
from fractions import Fraction

import numpy as np
import torch

import paper_2208_05683_gb300 as psf


def listed():
    return [
        # the smallest call: one exact 1-norm of a small operator, as a caller
        # checks or scales an input before an evaluation
        {"name": "norm1 grid 37x29", "call": "norm1", "matrix": "grid", "rows": 37, "cols": 29},
        # one product step by itself, unfiltered, with an addend and an identity
        # term: the building block that a caller composes other schemes from
        {"name": "product banded 30001", "call": "product", "matrix": "banded", "n": 30001, "w": 5, "w2": 17,
         "threshold": 0.0},
        # a small evaluation, where launches and latency count
        {"name": "exp lap1d 256", "call": "eval", "matrix": "lap1d", "n": 256, "norm": 2.0, "series": "exp",
         "tol": 1e-12, "option": ""},
        # the paper's banded N(0, 1) family at its own size and tolerance
        {"name": "cos normal 1000 w8", "call": "eval", "matrix": "normal", "n": 1000, "w": 8, "series": "cos",
         "tol": 1e-14, "option": ""},
        # the headline workload: exp of the operator on a 128 x 128 grid
        {"name": "exp grid 128x128", "call": "eval", "matrix": "grid", "rows": 128, "cols": 128, "norm": 4.0,
         "series": "exp", "tol": 1e-12, "option": ""},
        # an even series in W = Z^2 on a ragged grid
        {"name": "cos grid 101x97 square", "call": "eval", "matrix": "grid", "rows": 101, "cols": 97, "norm": 4.0,
         "series": "cos", "tol": 1e-12, "option": "square"},
        # a wide band of many short rows (the tolerance sweep's matrix)
        {"name": "exp banded 65536", "call": "eval", "matrix": "banded", "n": 65536, "w": 5, "norm": 2.0,
         "series": "exp", "tol": 1e-10, "option": ""},
        # large norms, many terms, the powers' norms estimated
        {"name": "exp normal 20000 w15 est", "call": "eval", "matrix": "normal", "n": 20000, "w": 15, "series": "exp",
         "tol": 1e-14, "option": "estimate"},
        # an unstructured matrix whose powers fill in: the late steps are dense
        {"name": "exp random 2000", "call": "eval", "matrix": "random", "n": 2000, "density": 0.01, "norm": 2.0,
         "series": "exp", "tol": 1e-12, "option": ""},
        # the largest grid: rows wider than any column window
        {"name": "exp grid 512x512", "call": "eval", "matrix": "grid", "rows": 512, "cols": 512, "norm": 4.0,
         "series": "exp", "tol": 1e-12, "option": ""},
        # many small instances in one call
        {"name": "batch 128", "call": "batch", "count": 128, "n_lo": 64, "n_hi": 4096, "series": "exp cosh",
         "tol": 1e-12},
        # a burst of mixed requests through the serving loop
        {"name": "serve 48", "call": "serve", "count": 48, "n_lo": 256, "n_hi": 16384, "series": "exp cos sinh",
         "tol": 1e-10},
    ]


def _spread(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["norm1", "product", "batch", "serve"] + ["eval"] * 8)
    if kind == "norm1":
        return {"call": "norm1", "matrix": "grid", "rows": _spread(rng, 8, 512), "cols": _spread(rng, 8, 512)}
    if kind == "product":
        return {"call": "product", "matrix": "banded", "n": _spread(rng, 200, 65536), "w": rng.randint(1, 12),
                "w2": rng.randint(1, 40), "threshold": rng.choice([0.0, 0.0, 1e-3, 0.1])}
    if kind == "batch":
        return {"call": "batch", "count": _spread(rng, 2, 128), "n_lo": 64, "n_hi": rng.randint(500, 4096),
                "series": rng.choice(["exp", "exp cosh"]), "tol": 1e-12}
    if kind == "serve":
        return {"call": "serve", "count": _spread(rng, 4, 48), "n_lo": 256, "n_hi": rng.randint(1000, 16384),
                "series": "exp cos sinh", "tol": rng.choice([1e-8, 1e-10, 1e-12])}
    matrix = rng.choice(["lap1d", "grid", "grid", "grid", "banded", "banded", "normal", "random"])
    c = {"call": "eval", "matrix": matrix}
    if matrix == "lap1d":
        c.update(n=_spread(rng, 64, 200000), norm=rng.uniform(1.0, 4.0))
    elif matrix == "grid":
        c.update(rows=_spread(rng, 12, 400), cols=_spread(rng, 12, 400), norm=rng.uniform(1.0, 4.0))
    elif matrix == "banded":
        c.update(n=_spread(rng, 300, 65536), w=rng.randint(2, 8), norm=rng.uniform(1.0, 4.0))
    elif matrix == "normal":
        c.update(n=_spread(rng, 300, 20000), w=rng.randint(1, 15))
    else:
        c.update(n=rng.randint(300, 2000), density=rng.uniform(0.002, 0.01), norm=rng.uniform(1.0, 2.0))
    c["series"] = rng.choice(["exp", "exp", "cos", "cosh", "sinh"])
    c["tol"] = 1e-14 if matrix == "normal" else rng.choice([1e-8, 1e-10, 1e-12, 1e-12])
    options = ["", "", "", "unfiltered", "estimate", "submult"] + (["square", "square"] if c["series"] != "exp" else [])
    # the submultiplicative bound and the unfiltered scheme are used on small norms and sparse powers
    if matrix in ("normal", "random") or c.get("rows", 1) * c.get("cols", 1) > 40000:
        options = [o for o in options if o not in ("unfiltered", "submult")]
    c["option"] = rng.choice(options)
    return c


# ---- inputs: CSR tensors on the GPU, the same bits for the same seed
def _generator(seed, salt):
    g = torch.Generator(device="cuda")
    g.manual_seed((int(seed) * 1000003 + salt) % (1 << 62))
    return g


def _uniform(g, *shape):
    return torch.rand(*shape, generator=g, device="cuda", dtype=torch.float64)


def _from_diagonals(n, offsets, vals, keep):
    """CSR of the n x n matrix with vals[i, d] at (i, i + offsets[d]) where keep[i, d]."""
    off = torch.tensor(offsets, device="cuda")
    col = torch.arange(n, device="cuda")[:, None] + off[None, :]
    keep = keep & (col >= 0) & (col < n)
    rowptr = torch.zeros(n + 1, dtype=torch.int32, device="cuda")
    rowptr[1:] = keep.sum(1).cumsum(0)
    return psf.DeviceCSR(n, rowptr, col[keep].to(torch.int32).contiguous(), vals[keep].contiguous())


def _scaled_symmetric(vals, keep, centre, norm):
    """Diagonal = -(row sum of |off-diagonals|), then scaled to a 1-norm (= the largest row sum)."""
    vals = torch.where(keep, vals, torch.zeros_like(vals))
    s = vals.abs().sum(1)
    vals[:, centre] = -s
    return vals * (norm / (2.0 * s).max())


def _grid(rows, cols, norm, g):
    """A five-point diffusion operator with edge conductances in [0.95, 1.05]."""
    n = rows * cols
    i = torch.arange(n, device="cuda")
    r, c = i // cols, i % cols
    east, south = 0.95 + 0.1 * _uniform(g, n), 0.95 + 0.1 * _uniform(g, n)
    keep = torch.stack([r > 0, c > 0, torch.ones_like(r, dtype=torch.bool), c < cols - 1, r < rows - 1], 1)
    vals = torch.stack([torch.roll(south, cols), torch.roll(east, 1), torch.zeros_like(east), east, south], 1)
    if cols == 1:
        keep[:, 1] = keep[:, 3] = False
    # Dirichlet edges: the diagonal counts the missing neighbours too
    vals = torch.where(keep, vals, torch.zeros_like(vals))
    vals[:, 2] = -(vals.sum(1) + (4 - (keep.sum(1) - 1)).to(torch.float64))
    if norm is not None:
        vals = vals * (norm / vals.abs().sum(1).max())
    return _from_diagonals(n, [-cols, -1, 0, 1, cols], vals, keep)


def _lap1d(n, norm, g):
    """The 1D operator of the same kind."""
    edge = 0.95 + 0.1 * _uniform(g, n)
    i = torch.arange(n, device="cuda")
    keep = torch.stack([i > 0, torch.ones_like(i, dtype=torch.bool), i < n - 1], 1)
    vals = torch.stack([torch.roll(edge, 1), torch.zeros_like(edge), edge], 1)
    vals = torch.where(keep, vals, torch.zeros_like(vals))
    vals[:, 1] = -(vals.sum(1) + (2 - (keep.sum(1) - 1)).to(torch.float64))
    return _from_diagonals(n, [-1, 0, 1], vals * (norm / vals.abs().sum(1).max()), keep)


def _banded(n, w, norm, g):
    """Symmetric, half-bandwidth w, off-diagonals U[-1, 1], diagonally balanced."""
    w = min(w, n - 1)
    up = 2.0 * _uniform(g, w, n) - 1.0
    offsets = list(range(-w, w + 1))
    i = torch.arange(n, device="cuda")
    cols = [torch.roll(up[-d - 1], -d) if d < 0 else up[d - 1] if d > 0 else torch.zeros_like(up[0]) for d in offsets]
    keep = torch.stack([(i + d >= 0) & (i + d < n) for d in offsets], 1)
    vals = _scaled_symmetric(torch.stack(cols, 1), keep, w, norm)
    return _from_diagonals(n, offsets, vals, keep)


def _normal(n, w, g):
    w = min(w, n - 1)
    vals = torch.randn(n, 2 * w + 1, generator=g, device="cuda", dtype=torch.float64)
    return _from_diagonals(n, list(range(-w, w + 1)), vals, torch.ones_like(vals, dtype=torch.bool))


def _random(n, density, norm, g):
    """Unstructured, entries U[-1, 1], scaled to a 1-norm."""
    d = 2.0 * _uniform(g, n, n) - 1.0
    d = torch.where(_uniform(g, n, n) < density, d, torch.zeros_like(d))
    d *= norm / d.abs().sum(0).max().clamp_min(1e-300)
    keep = d != 0
    rowptr = torch.zeros(n + 1, dtype=torch.int32, device="cuda")
    rowptr[1:] = keep.sum(1).cumsum(0)
    return psf.DeviceCSR(n, rowptr, keep.nonzero()[:, 1].to(torch.int32).contiguous(), d[keep].contiguous())


def _matrix(c, g):
    if c["matrix"] == "grid":
        return _grid(c["rows"], c["cols"], c.get("norm"), g)
    if c["matrix"] == "lap1d":
        return _lap1d(c["n"], c["norm"], g)
    if c["matrix"] == "banded":
        return _banded(c["n"], c["w"], c.get("norm", 2.0), g)
    if c["matrix"] == "normal":
        return _normal(c["n"], c["w"], g)
    return _random(c["n"], c["density"], c["norm"], g)


def _coeffs(kind):
    """Taylor coefficients, each the double nearest its exact value."""
    a = []
    for i in range(200):
        on = kind == "exp" or (i % 2 == (1 if kind == "sinh" else 0))
        sign = (-1) ** (i // 2) if kind == "cos" else 1
        a.append(float(Fraction(sign, math.factorial(i))) if on else 0.0)
    while a[-1] == 0.0:
        a.pop()
    return a


def _series(kind, tol, option=""):
    opts = {"": {}, "unfiltered": {"filtered": False}}.get(option, {option: True})
    return psf.Series(_coeffs(kind), tol, **opts)


def _instances(c):
    """The mixture's instances (matrix dict, series kind): sizes log-uniform, the same for every seed."""
    rng = random.Random(c["count"] * 7919 + c["n_lo"] * 31 + c["n_hi"])
    out = []
    for _ in range(c["count"]):
        n = _spread(rng, c["n_lo"], c["n_hi"])
        kind = rng.choice(["lap1d", "grid", "banded"])
        m = {"matrix": kind, "n": n, "w": 5, "norm": rng.uniform(1.0, 4.0)}
        if kind == "grid":
            m["rows"] = m["cols"] = max(2, int(round(math.sqrt(n))))
        out.append((m, rng.choice(c["series"].split())))
    return out


def _room(n, entries):
    """The caller's own result arrays, with room for as many entries as the case may give."""
    return [torch.zeros(n, dtype=torch.int32, device="cuda"), torch.zeros(entries, dtype=torch.int32, device="cuda"),
            torch.zeros(entries, dtype=torch.float64, device="cuda")]


def _entries(c, tol):
    """Room for a result: what the series' terms above the tolerance reach, or every term's reach when unfiltered."""
    n = c["rows"] * c["cols"] if c["matrix"] == "grid" else c["n"]
    terms, reach = _terms(c, tol)
    per_row = _row_len(c, terms if c.get("option") == "unfiltered" else 1.2 * reach + 2)
    return int(n * per_row) + 1


def prepare(case, seed):
    c = dict(case)
    g = _generator(seed, 17)
    if c["call"] in ("batch", "serve"):
        inst = _instances(c)
        # the mixtures share each kind's coefficients; every instance keeps its own series, as a server's clients do
        state = {"Z": [_matrix(m, g) for m, _ in inst], "series": [_series(k, c["tol"]) for _, k in inst]}
        state["out"] = _room(sum(z.n + 1 for z in state["Z"]), sum(_entries(m, c["tol"]) for m, _ in inst))
        if c["call"] == "serve":
            state["server"] = psf.Server(workers=4, max_batch=64)
    elif c["call"] == "product":
        state = {"A": _banded(c["n"], c["w"], 2.0, g), "B": _banded(c["n"], c["w2"], 1.0, g),
                 "M": _banded(c["n"], 3, 1.0, g), "threshold": c["threshold"]}
        if c["threshold"] > 0.0:
            state["out"] = _room(c["n"] + 1, c["n"] * min(c["n"], 2 * max(c["w"] + c["w2"], 3) + 1))
    else:
        state = {"Z": _matrix(c, g)}
        if c["call"] == "eval":
            state["series"] = _series(c["series"], c["tol"], c["option"])
            state["out"] = _room(state["Z"].n + 1, _entries(c, c["tol"]))
    state["call"] = c["call"]
    return state


def _into(out, ms):
    """The results, one after the other, in the caller's arrays (the rest of them stays 0)."""
    for buf, parts in zip(out, zip(*((m.rowptr, m.col, m.val) for m in ms))):
        to = buf[: sum(p.numel() for p in parts)]
        if len(parts) == 1:
            to.copy_(parts[0])
        else:
            torch.cat(parts, out=to)
    return out


def run(state):
    call = state["call"]
    if call == "norm1":
        return psf.norm1(state["Z"])
    if call == "product":
        c = psf.product_filter(state["A"], state["B"], [(0.5, state["M"]), (0.25, None)], threshold=state["threshold"]).csr
        return _into(state["out"], [c]) if "out" in state else [c.rowptr, c.col, c.val]
    if call == "eval":
        return _into(state["out"], [state["series"].eval(state["Z"]).csr])
    if call == "batch":
        return _into(state["out"], [r.csr for r in psf.eval_batch(state["series"], state["Z"])])
    server, done = state["server"], {}
    for tag, (s, z) in enumerate(zip(state["series"], state["Z"])):
        server.submit(s, z, tag)
    while len(done) < len(state["Z"]):
        for item in server.poll():
            done[item["tag"]] = item["result"].csr
    return _into(state["out"], [done[tag] for tag in range(len(state["Z"]))])


# ---- what a pass cannot do without
def _row_len(c, k):
    """Entries of a row of Z^k away from the edges."""
    if c["matrix"] == "grid":
        return min(2.0 * k * k + 2 * k + 1, float(c["rows"] * c["cols"]))
    if c["matrix"] == "random":
        return min(max(1.0, c["density"] * c["n"]) ** k, float(c["n"]))
    w = 1 if c["matrix"] == "lap1d" else c["w"]
    return min(2.0 * w * k + 1, float(c["n"]))


def _terms(c, tol):
    """The truncation length, and the power past which no entry of the result stays."""
    norm = c.get("norm") or 1.6 * c["w"] + 4.0
    terms = next(m for m in range(2, 200) if norm ** m / math.factorial(m) < tol / 2 and m > norm)
    reach = next(m for m in range(1, 200) if norm ** m / math.factorial(m) / 2.0 ** m < tol and 2 * m > norm)
    return terms, reach


def _eval_work(c, tol):
    """Bytes and flops of one evaluation: the products of the Paterson-Stockmeyer scheme of the truncated series
    (and of the powers' norms), the result's rows cut where the series' terms fall below the tolerance."""
    n = c["rows"] * c["cols"] if c["matrix"] == "grid" else c["n"]
    terms, reach = _terms(c, tol)
    q = max(1, math.isqrt(terms - 1))
    b = -(-terms // q)
    fma = 0.0
    if c.get("option") not in ("estimate", "submult"):
        fma += sum(_row_len(c, 1) * _row_len(c, k) for k in range(1, 10))
    else:
        fma += sum(_row_len(c, 1) * _row_len(c, k) for k in range(1, q))
    fma += sum(_row_len(c, q) * _row_len(c, min(reach, q * i)) for i in range(1, b))
    return {"bytes": 12.0 * n * (_row_len(c, 1) + _row_len(c, reach)) + 8.0 * n, "flops": 2.0 * n * fma}


def work(case):
    c = case
    if c["call"] in ("batch", "serve"):
        each = [_eval_work(m, c["tol"]) for m, _ in _instances(c)]
        return {k: sum(w[k] for w in each) for k in ("bytes", "flops")}
    if c["call"] == "norm1":
        n = c["rows"] * c["cols"]
        return {"bytes": 12.0 * 5 * n + 4.0 * n, "flops": 5.0 * n}
    if c["call"] == "product":
        a, b = 2.0 * c["w"] + 1, 2.0 * c["w2"] + 1
        return {"bytes": c["n"] * (12.0 * (a + b + 7 + a + b - 1) + 16.0), "flops": 2.0 * c["n"] * (a * b + 8)}
    return _eval_work(c, c["tol"])


def exact(case, seed):
    """Norms and unfiltered products have a value of their own; what a filtered evaluation keeps depends on
    the scheme's thresholds, entry by entry."""
    c = case
    if c["call"] == "norm1":
        z = prepare(case, seed)["Z"]
        col, val = z.col.cpu().numpy(), z.val.abs().cpu().numpy()
        return float(np.bincount(col, weights=val, minlength=z.n).max())
    if c["call"] == "product" and c["threshold"] == 0.0:
        s = prepare(case, seed)

        def rows(m, lo, hi):  # a block of rows, dense over the band that its columns span
            p0, p1 = int(m.rowptr[lo]), int(m.rowptr[hi])
            r = torch.repeat_interleave(torch.arange(hi - lo, device="cuda"), (m.rowptr[lo + 1:hi + 1] - m.rowptr[lo:hi]).long())
            return r, m.col[p0:p1].long(), m.val[p0:p1]

        n, w, out = c["n"], max(c["w"] + c["w2"], 3), []
        for lo in range(0, n, 1024):  # row blocks: the band keeps each block's columns together
            hi = min(n, lo + 1024)
            k0, k1 = max(0, lo - c["w"]), min(n, hi + c["w"])
            c0, c1 = max(0, lo - w), min(n, hi + w)
            a = torch.zeros(hi - lo, k1 - k0, dtype=torch.float64, device="cuda")
            b = torch.zeros(k1 - k0, c1 - c0, dtype=torch.float64, device="cuda")
            r, k, v = rows(s["A"], lo, hi)
            a[r, k - k0] = v
            r, k, v = rows(s["B"], k0, k1)
            b[r, k - c0] = v
            f = a @ b
            there = (a != 0).double() @ (b != 0).double() > 0
            r, k, v = rows(s["M"], lo, hi)
            f[r, k - c0] += 0.5 * v
            there[r, k - c0] = True
            i = torch.arange(hi - lo, device="cuda")
            f[i, i + lo - c0] += 0.25
            there[i, i + lo - c0] = True
            out.append(f[there])
        return [None, None, torch.cat(out)]
    return None
