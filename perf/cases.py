"""Performance cases: the work a user of this library has it do.

Every case is a dict with a ``kind``; ``prepare`` builds on the GPU what a
program holds before the call (matrices and vectors made from the seed, and
the prepared handles it keeps), ``run`` makes one pass through the public
entry points and returns everything the pass computes, ``work`` counts the
bytes and operations the pass cannot do without, and ``exact`` gives the
same outputs in plain 64-bit torch.

Kinds:
  spmv      y = A x with a matrix prepared once (a solver's inner loop)
  features  Table 1 features of a matrix that has just arrived
  onboard   a new matrix end to end: features, learned selection, prepare,
            first product
  cg        a conjugate-gradient solve (graph form), FP64 or mixed precision
  batch     many uneven matrices in one persistent launch
  host      y = A x with x and y in page-locked host memory
  train     one training step of the selector network

Matrices are square.  Families (the benchmark's): ``stencil`` (a 5-, 7- or
27-point stencil on an nx x ny x nz grid), ``random`` (``per_row`` uniform
columns a row), ``zipf`` (power-law row lengths, one very long row) and
``band`` (``per_row`` columns within a band around the diagonal).
"""
import math
import os

import numpy as np
import torch

import paper_1511_02494_gb300 as sp

DATA = os.path.join(os.path.dirname(os.path.abspath(sp.__file__)), "data")
VALUE_TYPES = {"f64": sp.VAL_F64, "f32": sp.VAL_F32, "bf16": sp.VAL_BF16}
H1, H2, K = 64, 64, 8          # the selector network's shape


def listed():
    return [
        # the parity-test matrix: the smallest call, where the launch counts
        dict(name="spmv_laplacian2d_64", kind="spmv", family="stencil", points=5, nx=64, ny=64, nz=1, values="f64"),
        # the benchmark's four bottleneck classes at its own sizes
        dict(name="spmv_stencil27_128", kind="spmv", family="stencil", points=27, nx=128, ny=128, nz=128, values="f64"),
        dict(name="spmv_random_4Mx16", kind="spmv", family="random", rows=1 << 22, per_row=16, values="f64"),
        dict(name="spmv_zipf_1M", kind="spmv", family="zipf", rows=1 << 20, alpha=1.8, max_len=200_000, values="f64"),
        dict(name="spmv_short_8M", kind="spmv", family="band", rows=1 << 23, per_row=2, band=16, values="f64"),
        # the features alone, on the rows that are hardest to split evenly
        dict(name="features_zipf_1M", kind="features", family="zipf", rows=1 << 20, alpha=1.8, max_len=200_000),
        # a new matrix: what the method costs before the first product is out
        dict(name="onboard_stencil27_100", kind="onboard", family="stencil", points=27, nx=100, ny=100, nz=100),
        # a small solve, where launches count, and the mixed-precision solve of the benchmark
        dict(name="cg_f64_33", kind="cg", nx=33, ny=33, nz=33, values="f64", iters=100, refine=0),
        dict(name="cg_bf16_128", kind="cg", nx=128, ny=128, nz=128, values="bf16", iters=100, refine=10),
        # the benchmark's batch
        dict(name="batch_512", kind="batch", count=512, lo=1e3, hi=1e5),
        # the benchmark's end-to-end form
        dict(name="host_stencil27_128", kind="host", family="stencil", points=27, nx=128, ny=128, nz=128),
        # a full-batch step at the training set's size
        dict(name="train_1600", kind="train", samples=1600),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_matrix(rng, rows_lo, rows_hi, max_nnz):
    family = rng.choice(("stencil", "random", "zipf", "band"))
    n = _log(rng, rows_lo, rows_hi)
    if family == "stencil":
        points = rng.choice((5, 7, 27))
        n = min(n, max_nnz // points)
        if points == 5:
            nx = max(2, int(round(math.sqrt(n) * math.exp(rng.uniform(-0.5, 0.5)))))
            return dict(family=family, points=points, nx=nx, ny=max(2, n // nx), nz=1)
        nx = max(2, int(round(n ** (1 / 3) * math.exp(rng.uniform(-0.4, 0.4)))))
        ny = max(2, int(round(math.sqrt(n / nx) * math.exp(rng.uniform(-0.4, 0.4)))))
        return dict(family=family, points=points, nx=nx, ny=ny, nz=max(2, n // (nx * ny)))
    if family == "random":
        per_row = rng.randint(2, 64)
        return dict(family=family, rows=min(n, max_nnz // per_row), per_row=per_row)
    if family == "zipf":
        alpha, longest = round(rng.uniform(1.5, 2.5), 3), max(2, min(n // 5, 200_000))
        n = min(n, int((max_nnz - longest) / _zipf_mean(alpha, longest)))
        return dict(family=family, rows=n, alpha=alpha, max_len=max(2, min(n // 5, longest)))
    return dict(family=family, rows=n, per_row=rng.randint(1, 4), band=rng.randint(5, 63))


def draw(rng):
    kind = rng.choice(("spmv", "spmv", "spmv", "features", "onboard", "cg", "batch", "host", "train"))
    if kind == "spmv":
        return dict(_draw_matrix(rng, 2_000, 6_000_000, 60_000_000), kind=kind,
                    values=rng.choice(("f64", "f64", "f32", "bf16")))
    if kind == "features":
        c = dict(_draw_matrix(rng, 10_000, 4_000_000, 28_000_000), kind=kind)
        if c["family"] == "stencil":
            c["holes"] = round(rng.uniform(0.01, 0.2), 3)   # couplings missing: a domain that does not fill its grid
        if c["family"] == "band":
            c["per_row"] = max(2, c["per_row"])
        return c
    if kind == "onboard":
        return dict(_draw_matrix(rng, 10_000, 2_000_000, 24_000_000), kind=kind)
    if kind == "host":
        return dict(_draw_matrix(rng, 10_000, 2_000_000, 50_000_000), kind=kind)
    if kind == "cg":
        values = rng.choice(("f64", "f64", "f32", "bf16"))
        side = _log(rng, 16, 120)
        return dict(kind=kind, nx=side, ny=max(2, side - rng.randint(0, 9)), nz=side + rng.randint(0, 7),
                    values=values, iters=rng.randint(40, 99), refine=0 if values == "f64" else rng.choice((5, 10, 20)))
    if kind == "batch":
        return dict(kind=kind, count=_log(rng, 8, 400), lo=1e3, hi=float(_log(rng, 1e4, 1e5)))
    return dict(kind=kind, samples=_log(rng, 100, 1600))


# ---- sizes known without the GPU -------------------------------------------------

def _zipf_mean(alpha, max_len):
    k = np.arange(1, max_len + 1, dtype=np.float64)
    w = k ** -alpha
    return float((k * w).sum() / w.sum())


def _size(c):
    """(rows, nonzeros) of a matrix; for the Zipf rows the expected count."""
    if c["family"] == "stencil":
        nx, ny, nz = c["nx"], c["ny"], c["nz"]
        n = nx * ny * nz
        if c["points"] == 27:
            nnz = (3 * nx - 2) * (3 * ny - 2) * (3 * nz - 2)
        else:
            nnz = n + 2 * ((nx - 1) * ny * nz + nx * (ny - 1) * nz + nx * ny * (nz - 1))
        return n, int(nnz * (1.0 - c.get("holes", 0.0)))
    if c["family"] == "zipf":
        return c["rows"], int(c["rows"] * _zipf_mean(c["alpha"], c["max_len"])) + c["max_len"]
    return c["rows"], c["rows"] * c["per_row"]


def _batch_specs(c):
    """The batch's matrices: rows spread over the logarithm of [lo, hi],
    families in turn, row lengths 2 to 200."""
    out = []
    for i in range(c["count"]):
        n = int(round(c["lo"] * (c["hi"] / c["lo"]) ** ((i * 0.6180339887498949 + 0.5) % 1.0)))
        r = (i * 0.7548776662466927 + 0.25) % 1.0
        if i % 4 == 0:
            m = max(4, round(n ** (1 / 3)))
            out.append(dict(family="stencil", points=27 if i % 8 == 0 else 7, nx=m, ny=m, nz=m))
        elif i % 4 == 1:
            out.append(dict(family="random", rows=n, per_row=2 + int(62 * r)))
        elif i % 4 == 2:
            out.append(dict(family="zipf", rows=n, alpha=1.5 + r, max_len=200))
        else:
            out.append(dict(family="band", rows=n, per_row=2 + int(3 * r), band=32))
    return out


# ---- matrices ------------------------------------------------------------------------

def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _uniform(n, g, lo=-1.0, hi=1.0):
    return lo + (hi - lo) * torch.rand(n, generator=g, dtype=torch.float64, device="cuda")


def _rowptr(lengths):
    rp = torch.zeros(lengths.numel() + 1, dtype=torch.int64, device="cuda")
    torch.cumsum(lengths, 0, out=rp[1:])
    return rp


def _sorted_columns(lengths, n_cols, g):
    """Per row its number of distinct increasing columns in [0, n_cols), uniform."""
    rows = torch.repeat_interleave(torch.arange(lengths.numel(), device="cuda"), lengths)
    span = (n_cols - lengths + 1)[rows]
    r = (torch.rand(rows.numel(), generator=g, dtype=torch.float64, device="cuda") * span).to(torch.int64)
    key = torch.sort(rows * (n_cols + 1) + torch.minimum(r, span - 1))[0]
    rank = torch.arange(rows.numel(), device="cuda") - _rowptr(lengths)[:-1][rows]
    return key - rows * (n_cols + 1) + rank, rows


def _stencil_pattern(c, holes=0.0, g=None):
    nx, ny, nz = c["nx"], c["ny"], c["nz"]
    reach = [(dz, dy, dx) for dz in (-1, 0, 1) for dy in (-1, 0, 1) for dx in (-1, 0, 1)]
    if c["points"] != 27:
        reach = [o for o in reach if sum(map(abs, o)) <= 1]
    if nz == 1:
        reach = [o for o in reach if o[0] == 0]
    i = torch.arange(nx * ny * nz, device="cuda")
    z, y, x = i // (ny * nx), i // nx % ny, i % nx
    cols, ok = [], []
    for dz, dy, dx in reach:
        cols.append(i + (dz * ny + dy) * nx + dx)
        ok.append((z + dz >= 0) & (z + dz < nz) & (y + dy >= 0) & (y + dy < ny) & (x + dx >= 0) & (x + dx < nx))
    ok = torch.stack(ok, 1)
    if holes:
        ok &= torch.rand(ok.shape, generator=g, device="cuda") >= holes
    return ok.sum(1), torch.stack(cols, 1)[ok]


def _matrix(c, seed):
    """The case's matrix with values ~U[-1, 1] (CSR on the GPU)."""
    g = _gen(seed)
    if c["family"] == "stencil":
        lengths, cols = _stencil_pattern(c, c.get("holes", 0.0), g)
    elif c["family"] == "random":
        lengths = torch.full((c["rows"],), c["per_row"], dtype=torch.int64, device="cuda")
        cols, _ = _sorted_columns(lengths, c["rows"], g)
    elif c["family"] == "zipf":
        k = torch.arange(1, c["max_len"] + 1, dtype=torch.float64, device="cuda")
        cdf = torch.cumsum(k.pow(-c["alpha"]), 0)
        u = torch.rand(c["rows"], generator=g, dtype=torch.float64, device="cuda")
        lengths = torch.clamp(torch.searchsorted(cdf / cdf[-1], u) + 1, 1, c["max_len"])
        lengths[torch.argmax(lengths)] = c["max_len"]
        cols, _ = _sorted_columns(lengths, c["rows"], g)
    else:
        width = min(c["band"], c["rows"])
        lengths = torch.full((c["rows"],), min(c["per_row"], width), dtype=torch.int64, device="cuda")
        cols, rows = _sorted_columns(lengths, width, g)
        cols = cols + torch.clamp(rows - width // 2, 0, c["rows"] - width)
    return _csr(lengths, cols, _uniform(cols.numel(), g))


def _csr(lengths, cols, val):
    n = lengths.numel()
    return sp.DeviceCSR(n, n, _rowptr(lengths).to(torch.int32), cols.to(torch.int32), val)


def _spd_matrix(c, seed):
    """7-point Laplacian with a coefficient ~U[0.5, 1.5] per edge and a
    strictly dominant diagonal (symmetric positive definite)."""
    lengths, cols = _stencil_pattern(dict(c, points=7))
    n = lengths.numel()
    rows = torch.repeat_interleave(torch.arange(n, device="cuda"), lengths)
    coef = _uniform(3 * n, _gen(seed), 0.5, 1.5).view(n, 3)
    d = (rows - cols).abs()
    axis = torch.where(d == 1, 0, torch.where(d == c["nx"], 1, 2))
    off = torch.where(d == 0, 0.0, -coef[torch.minimum(rows, cols), axis])
    # at most six terms a row, summed in a fixed order
    ends = _rowptr(lengths)
    diag = torch.ones(n, dtype=torch.float64, device="cuda")
    for k in range(7):
        has = lengths > k
        diag[has] += off[ends[:-1][has] + k].abs()
    return _csr(lengths, cols, torch.where(d == 0, diag[rows], off))


_models = []


def _selector():
    if not _models:
        _models.extend(sp.spmv_model_load(os.path.join(DATA, f))
                       for f in ("selector_mlp.bin", "selector_sliced_mlp.bin"))
    return _models


def _choice(A, values="f64"):
    if values != "f64":
        return sp.make_choice("sliced", value_type=VALUE_TYPES[values])
    return sp.spmv_select_model_refined(sp.spmv_features(A), *_selector())


def _empty(n):
    return torch.empty(n, dtype=torch.float64, device="cuda")


# ---- one case ------------------------------------------------------------------------

def prepare(case, seed):
    c, kind = case, case["kind"]
    if kind in ("spmv", "features", "onboard", "host"):
        A = _matrix(c, seed)
        x = _uniform(A.n_cols, _gen(seed + 1_000_003))
        s = dict(kind=kind, A=A, x=x, y=_empty(A.n_rows))
        if kind in ("spmv", "host"):
            s["P"] = sp.spmv_prepare(A, _choice(A, c.get("values", "f64")))
        if kind == "onboard":
            s["models"] = _selector()
        if kind == "host":
            s["xh"], s["yh"] = x.cpu().pin_memory(), torch.empty(A.n_rows, dtype=torch.float64).pin_memory()
        return s
    if kind == "cg":
        A = _spd_matrix(c, seed)
        exact = sp.spmv_prepare(A, sp.make_choice("sliced"))
        inner = exact if c["values"] == "f64" else \
            sp.spmv_prepare(A, sp.make_choice("sliced", value_type=VALUE_TYPES[c["values"]]))
        return dict(kind=kind, A=A, exact=exact, inner=inner, iters=c["iters"], refine=c["refine"],
                    b=_uniform(A.n_rows, _gen(seed + 1_000_003)), x=_empty(A.n_rows), resid=_empty(c["iters"] + 1))
    if kind == "batch":
        mats = [_matrix(m, seed * 1009 + i) for i, m in enumerate(_batch_specs(c))]
        x = _uniform(sum(A.n_cols for A in mats), _gen(seed + 1_000_003))
        y = _empty(sum(A.n_rows for A in mats))
        preps = [sp.spmv_prepare(A, sp.make_choice("sliced"), trusted=True) for A in mats]
        B = sp.spmv_batch_create_sliced(preps)
        sp.spmv_batch_bind(B, x.split([A.n_cols for A in mats]), y.split([A.n_rows for A in mats]))
        return dict(kind=kind, mats=mats, B=B, x=x, y=y)
    return dict(_train_state(c, seed), kind=kind)


def _train_state(c, seed):
    """A network in mid-training: standardised features, cost-sensitive
    targets, and moments of the size a few hundred steps leave."""
    g = _gen(seed)
    n = c["samples"]

    def normal(*shape):
        return torch.randn(*shape, generator=g, dtype=torch.float32, device="cuda")
    p = torch.cat([w for i, o in ((16, H1), (H1, H2), (H2, K))
                   for w in (normal(o * i) * math.sqrt(2.0 / i), 0.1 * normal(o))])
    q = torch.softmax(4.0 * normal(n, K), 1)
    return dict(z=normal(n, 16), q=q, p=p, g=torch.zeros_like(p), m=1e-3 * normal(p.numel()),
                v=1e-6 * (0.1 + torch.rand(p.numel(), generator=g, dtype=torch.float32, device="cuda")),
                loss=torch.zeros(1, dtype=torch.float32, device="cuda"), step=300)


def run(s):
    kind = s["kind"]
    if kind == "spmv":
        sp.spmv(s["P"], s["x"], s["y"])
        return s["y"]
    if kind == "features":
        return _features_out(sp.spmv_features(s["A"]))
    if kind == "onboard":
        f = sp.spmv_features(s["A"])
        ch = sp.spmv_select_model_refined(f, *s["models"])
        s["P"] = sp.spmv_prepare(s["A"], ch)
        sp.spmv(s["P"], s["x"], s["y"])
        return {"y": s["y"], "features": _features_out(f),
                "choice": np.array([ch.variant, ch.threads_per_row, ch.block_nnz, ch.items_per_warp])}
    if kind == "cg":
        s["x"].zero_()
        sp.spmv_cg(s["inner"], s["b"], s["x"], s["iters"], s["refine"], A_exact=s["exact"], resid=s["resid"],
                   use_graph=True)
        return s["x"], s["resid"]
    if kind == "batch":
        sp.spmv_batch_run(s["B"], use_graph=True)
        return s["y"]
    if kind == "host":
        sp.spmv_host(s["P"], s["xh"], s["yh"])
        return s["yh"]
    s["step"] += 1
    sp.spmv_mlp_loss_grad_soft(s["p"], H1, H2, K, s["z"], s["q"], s["g"], s["loss"])
    sp.spmv_mlp_adam(s["p"], s["g"], s["m"], s["v"], s["step"], lr=3e-3, weight_decay=1e-4)
    return {k: s[k] for k in ("loss", "g", "p", "m", "v")}


RATIOS = ("density", "nnz_avg", "nnz_sd", "bw_avg", "bw_sd", "disp_avg", "disp_sd", "clustering", "miss_ratio")
COUNTS = ("n_rows", "n_cols", "nnz", "line_bytes", "working_set_bytes", "nnz_min", "nnz_max", "nnz_sum",
          "nnz_sumsq_lo", "nnz_sumsq_hi", "bw_min", "bw_max", "bw_sum", "bw_sumsq_lo", "bw_sumsq_hi", "disp_sum",
          "disp_sumsq_lo", "disp_sumsq_hi", "clust_sum", "ngroups_sum", "misses_sum")


def _features_out(f):
    return {"counts": np.array([getattr(f, k) for k in COUNTS], dtype=np.uint64).view(np.int64),
            "ratios": np.array([getattr(f, k) for k in RATIOS]), "vec": np.array(f.vec, dtype=np.float32)}


# ---- what a pass cannot do without ---------------------------------------------------

def work(case):
    c, kind = case, case["kind"]
    if kind in ("spmv", "features", "onboard", "host"):
        n, nnz = _size(c)
        if kind == "features":
            return {"bytes": 4 * (n + 1) + 4 * nnz, "flops": 0}
        vb = {"f64": 8, "f32": 4, "bf16": 2}[c.get("values", "f64")]
        once = (vb + 4) * nnz + 4 * (n + 1) + 16 * n
        # a new matrix: also its prepared form, written once
        return {"bytes": once + (12 * nnz if kind == "onboard" else 0), "flops": 2 * nnz}
    if kind == "cg":
        n, nnz = _size(dict(c, family="stencil", points=7))
        vb = {"f64": 8, "f32": 4, "bf16": 2}[c["values"]]
        # per iteration the operator once, x, r and p read and written, q written and read
        exact = c["iters"] // c["refine"] if c["refine"] else 0
        return {"bytes": c["iters"] * ((vb + 4) * nnz + 64 * n) + exact * (12 * nnz + 16 * n),
                "flops": (c["iters"] + exact) * 2 * nnz + c["iters"] * 10 * n}
    if kind == "batch":
        sizes = [_size(m) for m in _batch_specs(c)]
        return {"bytes": sum(12 * nnz + 4 * (n + 1) + 16 * n for n, nnz in sizes), "flops": 2 * sum(z for _, z in sizes)}
    n, params = c["samples"], 16 * H1 + H1 + H1 * H2 + H2 + H2 * K + K
    return {"bytes": 4 * n * (16 + K) + 4 * params * 8, "flops": 6 * n * params}


# ---- the same outputs in plain 64-bit torch ---------------------------------------------

def _times(A, x, val=None):
    rows = torch.repeat_interleave(torch.arange(A.n_rows, device="cuda"), (A.rowptr[1:] - A.rowptr[:-1]).long())
    return torch.zeros_like(x).index_add_(0, rows, (A.val if val is None else val) * x[A.colind.long()])


def _stored(val, values):
    return val if values == "f64" else val.to({"f32": torch.float32, "bf16": torch.bfloat16}[values]).double()


def exact(case, seed):
    c, kind = case, case["kind"]
    if kind in ("spmv", "onboard", "host"):
        A = _matrix(c, seed)
        y = _times(A, _uniform(A.n_cols, _gen(seed + 1_000_003)), _stored(A.val, c.get("values", "f64")))
        if kind == "onboard":
            return {"y": y, "features": _exact_features(A), "choice": None}
        return y.cpu() if kind == "host" else y
    if kind == "features":
        return _exact_features(_matrix(c, seed))
    if kind == "cg":
        return _exact_cg(c, seed)
    if kind == "batch":
        mats = [_matrix(m, seed * 1009 + i) for i, m in enumerate(_batch_specs(c))]
        xs = _uniform(sum(A.n_cols for A in mats), _gen(seed + 1_000_003)).split([A.n_cols for A in mats])
        return torch.cat([_times(A, x) for A, x in zip(mats, xs)])
    return _exact_step(_train_state(c, seed))


def _exact_features(A):
    n, nnz = A.n_rows, A.nnz
    rp, ci = A.rowptr.long(), A.colind.long()
    length = rp[1:] - rp[:-1]
    rows = torch.repeat_interleave(torch.arange(n, device="cuda"), length)
    first, last = ci[rp[:-1].clamp(max=nnz - 1)], ci[(rp[1:] - 1).clamp(min=0)]
    gap = torch.zeros_like(ci)
    gap[1:] = ci[1:] - ci[:-1]
    inner = torch.ones(nnz, dtype=torch.bool, device="cuda")
    inner[rp[:-1][length > 0]] = False
    full = length > 0

    def per_row(mark):
        return torch.zeros(n, dtype=torch.float64, device="cuda").index_add_(0, rows, mark.double()) + full
    groups, misses = per_row(inner & (gap != 1)), per_row(inner & (8 * gap > 128))
    bw = torch.where(full, last - first, 0).double()
    ln = length.double()
    disp = torch.where(full, ln / (bw + 1), 0.0)
    clust = torch.where(full, groups / ln.clamp(min=1), 0.0)
    mean, sd = (lambda v: v.mean().item()), (lambda v: v.std(correction=0).item())
    density = nnz / (n * A.n_cols)
    r = [density, mean(ln), sd(ln), mean(bw), sd(bw), mean(disp), sd(disp), mean(clust), mean(misses)]
    fits = 4 * (n + 1) + 12 * nnz + 16 * n <= torch.cuda.get_device_properties(0).L2_cache_size

    def lg(v):
        return math.log2(1.0 + v)
    vec = [float(fits), math.log2(max(density, 2.0 ** -64)), lg(ln.min().item()), lg(ln.max().item()), lg(r[1]), lg(r[2]),
           lg(bw.min().item()), lg(bw.max().item()), lg(r[3]), lg(r[4]), r[5], r[6], r[7], lg(r[8]), lg(n), lg(nnz)]
    return {"counts": None, "ratios": np.array(r), "vec": np.array(vec)}


def _exact_cg(c, seed):
    A = _spd_matrix(c, seed)
    b = _uniform(A.n_rows, _gen(seed + 1_000_003))
    val = _stored(A.val, c["values"])
    x, r, p = torch.zeros_like(b), b.clone(), b.clone()
    rs = torch.dot(r, r)
    resid = [rs.sqrt()]
    for t in range(1, c["iters"] + 1):
        q = _times(A, p, val)
        alpha = rs / torch.dot(p, q)
        x = x + alpha * p
        restart = c["refine"] and t % c["refine"] == 0
        r = b - _times(A, x) if restart else r - alpha * q
        rs, old = torch.dot(r, r), rs
        p = r.clone() if restart else r + (rs / old) * p
        resid.append(rs.sqrt())
    return x, torch.stack(resid)


def _exact_step(s):
    p = s["p"].double().requires_grad_()
    at, w = 0, []
    for size in (16 * H1, H1, H1 * H2, H2, H2 * K, K):
        w.append(p[at:at + size])
        at += size
    a = torch.relu(s["z"].double() @ w[0].view(H1, 16).T + w[1])
    a = torch.relu(a @ w[2].view(H2, H1).T + w[3])
    loss = -(s["q"].double() * torch.log_softmax(a @ w[4].view(K, H2).T + w[5], 1)).sum(1).mean()
    loss.backward()
    g, step = p.grad, s["step"] + 1
    m = 0.9 * s["m"].double() + 0.1 * g
    v = 0.999 * s["v"].double() + 0.001 * g * g
    new = s["p"].double()
    new = new - 3e-3 * (m / (1 - 0.9 ** step) / ((v / (1 - 0.999 ** step)).sqrt() + 1e-8) + 1e-4 * new)
    return {"loss": loss.detach().view(1), "g": g, "p": new, "m": m, "v": v}
