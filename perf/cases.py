"""The work this library is measured on: calls of its public entry points as a
user's program makes them, over the sizes, types and layouts the entry points
serve (listed()), more of the same ranges (draw()), inputs (prepare()), one pass
(run()), what a pass cannot do without (work()), and the same results from plain
torch in 64 bits (exact()).

Every case has a "kind" (which program it is), a storage type "dtype" and sizes.
All inputs are drawn on the device from the seed.
"""
from __future__ import annotations

import math

import torch

import paper_1409_0669_gb300 as lak
from paper_1409_0669_gb300 import autograd as lak_autograd
from paper_1409_0669_gb300 import batch as lak_batch

DTYPES = {"f32": torch.float32, "f64": torch.float64, "bf16": torch.bfloat16,
          "f16": torch.float16}
ESIZE = {"f32": 4, "f64": 8, "bf16": 2, "f16": 2}
DEV = "cuda"


# ---- the cases -------------------------------------------------------------------

def listed():
    return [
        # The smallest calls: one step of a small 2D problem -- update, inner
        # product, 5-point Laplacian product and a 1024^2 dense product, each a few
        # microseconds of GPU work, so call overhead and launches count.
        {"name": "small_step_f32", "kind": "small", "dtype": "f32", "grid": 256, "order": 1024},
        # Long vectors: the update, the inner product and the compensated inner
        # product on the largest vectors of the size sweep (pure streaming).
        {"name": "vectors_f32", "kind": "vectors", "dtype": "f32", "n": 100_000_000},
        # Shifted slices of one signal: first difference s[1:] - s[:-1] and the
        # lag-1 autocorrelation; the operands never share their alignment.
        {"name": "lagged_bf16", "kind": "lagged", "dtype": "bf16", "n": 21_544_347, "lag": 1},
        # A dense product with ragged sizes: odd row length, so every row starts
        # at another offset (16-bit storage, row-major).
        {"name": "gemv_ragged_bf16", "kind": "gemv", "dtype": "bf16", "m": 12_007, "n": 11_003},
        # Gram-Schmidt of a Krylov solver: projections h = V w on 30 basis vectors
        # of a 3D grid (few, very long rows), w - V^T h (the same storage the other
        # way round: very many, very short rows), and its norm.
        {"name": "orthogonalise_f64", "kind": "ortho", "dtype": "f64", "k": 30, "n": 2_097_152},
        # One Chebyshev iteration on a 3D Poisson problem: stencil product, residual
        # with its norm, search direction, solution (coefficients known beforehand,
        # so nothing is read back).
        {"name": "chebyshev_f64", "kind": "chebyshev", "dtype": "f64", "grid": 128},
        # Sparse product with random columns and power-law row lengths (a graph).
        {"name": "spmv_graph_f64", "kind": "spmv", "dtype": "f64", "matrix": "powerlaw",
         "size": 2_000_000},
        # Sparse product of a 3D elasticity matrix: rows of up to 81 entries, three
        # unknowns per node, 27 neighbours.
        {"name": "spmv_elastic_f64", "kind": "spmv", "dtype": "f64", "matrix": "elastic",
         "size": 56},
        # 4096 uneven dense products in one persistent launch, planned once.
        {"name": "batch_gemv_bf16", "kind": "batch_gemv", "dtype": "bf16", "count": 4096},
        # 1024 uneven sparse products in one persistent launch, planned once.
        {"name": "batch_spmv_f32", "kind": "batch_spmv", "dtype": "f32", "count": 1024},
        # Training, dense: loss <A x, t>, its gradients with respect to A, x and t.
        {"name": "grad_dense_f32", "kind": "grad_dense", "dtype": "f32", "m": 5000, "n": 3001},
        # Training, sparse, on a graph that is new in every step: forward and
        # backward of y = A x, the pattern's transpose made on the way.
        {"name": "grad_sparse_f32", "kind": "grad_sparse", "dtype": "f32", "matrix": "powerlaw",
         "size": 2_000_000},
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    """One more case of the listed ones' ranges."""
    kind = rng.choice(["small", "vectors", "lagged", "gemv", "ortho", "chebyshev", "spmv", "spmv",
                       "batch_gemv", "batch_spmv", "grad_dense", "grad_sparse"])
    c = {"kind": kind, "dtype": rng.choice(["f32", "f64", "bf16", "f16"])}
    if kind == "small":
        c.update(grid=rng.randint(96, 400), order=rng.randint(512, 1500))
    elif kind == "vectors":
        c["dtype"] = rng.choice(["f32", "bf16", "f16"])       # what the compensated form takes
        c["n"] = _log_int(rng, 1000, 100_000_000)
    elif kind == "lagged":
        c.update(n=_log_int(rng, 1000, 100_000_000), lag=rng.randint(1, 64))
    elif kind == "gemv":
        c.update(m=_log_int(rng, 64, 16_384), n=_log_int(rng, 64, 16_384))
    elif kind == "ortho":
        c["dtype"] = rng.choice(["f32", "f64"])
        c.update(k=rng.randint(2, 64), n=_log_int(rng, 10_000, 4_000_000))
    elif kind == "chebyshev":
        c["dtype"] = rng.choice(["f32", "f64"])
        c["grid"] = _log_int(rng, 16, 200)
    elif kind == "spmv":
        _draw_matrix(rng, c)
    elif kind == "batch_gemv":
        c["count"] = _log_int(rng, 64, 4096 if ESIZE[c["dtype"]] == 2 else 1024)
    elif kind == "batch_spmv":
        c["count"] = _log_int(rng, 64, 1024 if ESIZE[c["dtype"]] < 8 else 512)
    elif kind == "grad_dense":
        c["dtype"] = rng.choice(["f32", "f64"])
        c.update(m=_log_int(rng, 100, 8000), n=_log_int(rng, 100, 8000))
    else:
        c["dtype"] = rng.choice(["f32", "f64"])
        _draw_matrix(rng, c)
    return c


def _draw_matrix(rng, c):
    c["matrix"] = rng.choice(["powerlaw", "elastic", "laplace"])
    if c["matrix"] == "powerlaw":
        c["size"] = _log_int(rng, 1000, 2_000_000)
    elif c["matrix"] == "elastic":
        c["size"] = _log_int(rng, 8, 56)
    else:
        c["size"] = _log_int(rng, 16, 160)


# ---- inputs ------------------------------------------------------------------------

def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(seed)


def _uniform(g, n, dtype, lo=-1.0, hi=1.0):
    if dtype in (torch.float32, torch.float64):
        return torch.empty(n, dtype=dtype, device=DEV).uniform_(lo, hi, generator=g)
    return torch.empty(n, dtype=torch.float32, device=DEV).uniform_(lo, hi, generator=g).to(dtype)


def _mixed(g, n, dtype):
    """Random signs, magnitudes log-uniform in 1e-4 .. 1e4."""
    e = torch.empty(n, dtype=torch.float32, device=DEV).uniform_(-4.0, 4.0, generator=g)
    sign = torch.empty(n, dtype=torch.float32, device=DEV).uniform_(-1.0, 1.0, generator=g).sign()
    return (sign * torch.pow(10.0, e)).to(dtype)


def _grid_csr(n, reach, dofs):
    """Pattern of an n^3 grid, every node coupled to the neighbours for which
    `reach(dx, dy, dz)` holds, `dofs` unknowns per node: (row_ptr, col_idx) int32,
    columns sorted."""
    p = torch.arange(n ** 3, device=DEV)
    i, j, k = p % n, (p // n) % n, p // (n * n)
    cols, mask = [], []
    for dz in (-1, 0, 1):
        for dy in (-1, 0, 1):
            for dx in (-1, 0, 1):
                if not reach(dx, dy, dz):
                    continue
                cols.append(p + (dz * n + dy) * n + dx)
                mask.append((i + dx >= 0) & (i + dx < n) & (j + dy >= 0) & (j + dy < n)
                            & (k + dz >= 0) & (k + dz < n))
    mask = torch.stack(mask, 1)
    counts = (mask.sum(1) * dofs).repeat_interleave(dofs)
    cols = torch.stack(cols, 1).to(torch.int32)
    if dofs > 1:
        b = torch.arange(dofs, device=DEV, dtype=torch.int32)
        cols = (cols[:, :, None] * dofs + b).reshape(len(p), 1, -1).expand(-1, dofs, -1)
        mask = mask[:, :, None].expand(-1, -1, dofs).reshape(len(p), 1, -1).expand(-1, dofs, -1)
    rp = torch.zeros(len(counts) + 1, dtype=torch.int32, device=DEV)
    rp[1:] = torch.cumsum(counts, 0)
    return rp, cols[mask].contiguous()


def _powerlaw_lengths():
    """P(k) ~ k^-a on 4 .. 256 with mean 16."""
    k = torch.arange(4, 257, dtype=torch.float64, device=DEV)
    w = k ** -1.9647
    return k.to(torch.int32), w / w.sum()


def _csr(c, seed, dtype):
    """(row_ptr, col_idx, vals, n_cols) of the case's matrix."""
    g = _gen(seed)
    if c["matrix"] == "powerlaw":
        m = c["size"]
        k, w = _powerlaw_lengths()                       # row lengths go by the size alone
        lens = k[torch.multinomial(w, m, replacement=True, generator=_gen(m))].clamp(max=m)
        rp = torch.zeros(m + 1, dtype=torch.int32, device=DEV)
        rp[1:] = torch.cumsum(lens, 0)
        nnz = int(rp[-1])
        key = torch.randint(0, m, (nnz,), generator=g, device=DEV)
        key += torch.arange(m, device=DEV).repeat_interleave(lens.long()) * m
        key = key.sort()[0].remainder_(m)                # sorted columns in every row
        ci = key.to(torch.int32)
    elif c["matrix"] == "elastic":
        s = c["size"]
        m = 3 * s ** 3
        rp, ci = _grid_csr(s, lambda dx, dy, dz: True, 3)
    else:
        s = c["size"]
        m = s ** 3
        rp, ci = _grid_csr(s, lambda dx, dy, dz: abs(dx) + abs(dy) + abs(dz) <= 1, 1)
        rows = torch.arange(m, device=DEV).repeat_interleave((rp[1:] - rp[:-1]).long())
        return rp, ci, torch.where(rows == ci, 6.0, -1.0).to(dtype), m
    vals = torch.randn(ci.numel(), generator=g, device=DEV, dtype=torch.float32).to(dtype)
    return rp, ci, vals, m


def _laplace2d(n, dtype):
    p = torch.arange(n * n, device=DEV)
    i, j = p % n, p // n
    offs = torch.tensor([-n, -1, 0, 1, n], device=DEV)
    mask = torch.stack([j > 0, i > 0, i >= 0, i < n - 1, j < n - 1], 1)
    rp = torch.zeros(n * n + 1, dtype=torch.int32, device=DEV)
    rp[1:] = torch.cumsum(mask.sum(1), 0)
    ci = (p[:, None] + offs)[mask].to(torch.int32)
    v = torch.where(offs == 0, 4.0, -1.0).expand(n * n, 5)[mask].to(dtype)
    return rp, ci, v


def _flat_slices(sizes, align=64):
    """Starts of slices of the given sizes in one buffer, each on an `align` boundary."""
    starts, o = [], 0
    for s in sizes:
        starts.append(o)
        o += -(-s // align) * align
    return starts, o


def _sizes(seed, count, lo, hi):
    """`count` log-uniform sizes (instance sizes go by the case alone)."""
    g = torch.Generator().manual_seed(seed)
    u = torch.rand(count, generator=g, dtype=torch.float64)
    return [int(v) for v in torch.exp(math.log(lo) + u * math.log((hi + 1) / lo)).floor().clamp(lo, hi)]


def _acc(dtype):
    return torch.float64 if dtype == torch.float64 else torch.float32


def prepare(case, seed):
    kind, dt = case["kind"], DTYPES[case["dtype"]]
    g = _gen(seed)
    s = {"kind": kind, "dtype": dt}
    if kind == "small":
        n, o = case["grid"] ** 2, case["order"]
        s["y"], s["z"] = _uniform(g, n, dt), _uniform(g, n, dt)
        s["csr"] = _laplace2d(case["grid"], dt)
        s["A"] = torch.randn(o, o, generator=g, device=DEV, dtype=torch.float32).to(dt)
        s["v"] = _uniform(g, o, dt)
        s["x"], s["q"], s["b"] = (torch.empty(k, dtype=dt, device=DEV) for k in (n, n, o))
        s["dot"] = torch.empty(1, dtype=_acc(dt), device=DEV)
    elif kind == "vectors":
        n = case["n"]
        s["y"], s["z"] = _uniform(g, n, dt), _uniform(g, n, dt)
        # magnitudes far apart; FP16 holds 1e-4 .. 1e4 too
        s["p"], s["q"] = _mixed(g, n, dt), _mixed(g, n, dt)
        s["x"] = torch.empty(n, dtype=dt, device=DEV)
        s["dot"] = torch.empty(1, dtype=_acc(dt), device=DEV)
        s["cdot"] = torch.empty(1, dtype=torch.float64, device=DEV)
    elif kind == "lagged":
        n, lag = case["n"], case["lag"]
        signal = _uniform(g, n + lag, dt, 0.0, 1.0)           # intensities
        s["late"], s["early"] = signal[lag:], signal[:n]
        s["x"] = torch.empty(n, dtype=dt, device=DEV)
        s["dot"] = torch.empty(1, dtype=_acc(dt), device=DEV)
    elif kind == "gemv":
        m, n = case["m"], case["n"]
        if dt == torch.float64:
            s["A"] = torch.randn(m, n, generator=g, device=DEV, dtype=dt)
        else:
            s["A"] = torch.randn(m, n, generator=g, device=DEV, dtype=torch.float32).to(dt)
        s["x"] = _uniform(g, n, dt)
        s["y"] = torch.empty(m, dtype=dt, device=DEV)
    elif kind == "ortho":
        k, n = case["k"], case["n"]
        s["V"] = torch.randn(k, n, generator=g, device=DEV, dtype=dt).div_(math.sqrt(n))
        s["w"] = torch.randn(n, generator=g, device=DEV, dtype=dt)
        s["w"] += s["V"].sum(0) * math.sqrt(n)                # projections worth removing
        s["h"] = torch.empty(k, dtype=dt, device=DEV)
        s["r"] = torch.empty(n, dtype=dt, device=DEV)
        s["nrm"] = torch.empty(1, dtype=dt, device=DEV)
    elif kind == "chebyshev":
        n = case["grid"] ** 3
        s["csr"] = _csr({"matrix": "laplace", "size": case["grid"]}, seed, dt)
        s["d"], s["r"], s["u"] = (_uniform(g, n, dt) for _ in range(3))
        s["q"], s["r2"], s["d2"], s["u2"] = (torch.empty(n, dtype=dt, device=DEV) for _ in range(4))
        s["nrm"] = torch.empty(1, dtype=dt, device=DEV)
    elif kind == "spmv":
        s["csr"] = _csr(case, seed, dt)
        s["x"] = _uniform(g, s["csr"][3], dt)
        s["y"] = torch.empty(s["csr"][0].numel() - 1, dtype=dt, device=DEV)
    elif kind == "batch_gemv":
        ms, ns = _sizes(3, case["count"], 64, 4096), _sizes(4, case["count"], 64, 4096)
        oa, ta = _flat_slices([m * n for m, n in zip(ms, ns)])
        ox, tx = _flat_slices(ns)
        oy, ty = _flat_slices(ms)
        draw_dt = torch.float32 if dt == torch.float16 else dt
        A = torch.empty(ta, dtype=dt, device=DEV)
        for o in range(0, ta, 1 << 30):
            part = A[o:o + (1 << 30)]
            part.copy_(torch.randn(part.numel(), generator=g, device=DEV, dtype=draw_dt))
        x = _uniform(g, tx, dt)
        s["y"] = torch.zeros(ty, dtype=dt, device=DEV)
        s["As"] = [A[o:o + m * n].view(m, n) for o, m, n in zip(oa, ms, ns)]
        s["xs"] = [x[o:o + n] for o, n in zip(ox, ns)]
        s["ys"] = [s["y"][o:o + m] for o, m in zip(oy, ms)]
        s["batch"] = lak_batch.gemv_batch(s["As"], s["xs"], s["ys"])
    elif kind == "batch_spmv":
        ms = _sizes(5, case["count"], 1000, 200_000)
        lens = torch.randint(5, 65, (sum(ms),), generator=g, device=DEV, dtype=torch.int32)
        lens[torch.tensor(ms, device=DEV).cumsum(0) - 1] = 33
        first = torch.cumsum(lens, 0)                         # entries up to and with a row
        ends = first[torch.tensor(ms, device=DEV).cumsum(0) - 1].tolist()
        nnzs = [b - a for a, b in zip([0] + ends, ends)]
        oe, te = _flat_slices(nnzs)
        orp, trp = _flat_slices([m + 1 for m in ms])
        ov, tv = _flat_slices(ms)
        rp = torch.zeros(trp, dtype=torch.int32, device=DEV)
        ci = torch.empty(te, dtype=torch.int32, device=DEV)
        vals = torch.empty(te, dtype=dt, device=DEV)
        for o in range(0, te, 1 << 28):
            part = vals[o:o + (1 << 28)]
            part.copy_(torch.randn(part.numel(), generator=g, device=DEV, dtype=torch.float32))
        x = _uniform(g, tv, dt)
        s["y"] = torch.zeros(tv, dtype=dt, device=DEV)
        s["csrs"], row, before = [], 0, 0
        for m, nnz, a, b, end in zip(ms, nnzs, orp, oe, ends):
            rp[a + 1:a + m + 1] = first[row:row + m] - before
            torch.randint(0, m, (nnz,), generator=g, device=DEV, out=ci[b:b + nnz])
            s["csrs"].append((rp[a:a + m + 1], ci[b:b + nnz], vals[b:b + nnz], m))
            row, before = row + m, end
        s["xs"] = [x[o:o + m] for o, m in zip(ov, ms)]
        s["ys"] = [s["y"][o:o + m] for o, m in zip(ov, ms)]
        s["batch"] = lak_batch.spmv_batch(s["csrs"], s["xs"], s["ys"])
    elif kind == "grad_dense":
        m, n = case["m"], case["n"]
        s["A"] = torch.randn(m, n, generator=g, device=DEV, dtype=dt).requires_grad_()
        s["x"] = _uniform(g, n, dt).requires_grad_()
        t = s["A"].detach() @ s["x"].detach()                 # a target near the output
        s["t"] = (t + 0.5 * torch.randn(m, generator=g, device=DEV, dtype=dt)).requires_grad_()
    elif kind == "grad_sparse":
        rp, ci, vals, n = _csr(case, seed, dt)
        s["rp"], s["ci"], s["n"] = rp, ci, n
        s["vals"] = vals.requires_grad_()
        s["x"] = _uniform(g, n, dt).requires_grad_()
        s["dy"] = _uniform(g, rp.numel() - 1, dt)
    else:
        raise ValueError(kind)
    return s


# ---- one pass ----------------------------------------------------------------------

CHEB = (0.37, 0.21)            # coefficients of one Chebyshev step


def run(s):
    kind = s["kind"]
    if kind == "small":
        rp, ci, v = s["csr"]
        lak.vec_axpy(s["x"], s["y"], s["z"], 0.5)
        lak.vec_dot(s["x"], s["y"], out=s["dot"])
        lak.csr_spmv(rp, ci, v, s["x"], y=s["q"])
        lak.dense_gemv(s["A"], s["v"], y=s["b"])
        return {"x": s["x"], "dot": s["dot"], "q": s["q"], "b": s["b"]}
    if kind == "vectors":
        lak.vec_axpy(s["x"], s["y"], s["z"], 0.5)
        lak.vec_dot(s["x"], s["y"], out=s["dot"])
        lak.vec_dot_compensated(s["p"], s["q"], out=s["cdot"])
        return {"x": s["x"], "dot": s["dot"], "cdot": s["cdot"]}
    if kind == "lagged":
        lak.vec_axpy(s["x"], s["late"], s["early"], -1.0)
        lak.vec_dot(s["late"], s["early"], out=s["dot"])
        return {"x": s["x"], "dot": s["dot"]}
    if kind == "gemv":
        lak.dense_gemv(s["A"], s["x"], y=s["y"])
        return {"y": s["y"]}
    if kind == "ortho":
        lak.dense_gemv(s["V"], s["w"], y=s["h"])
        lak.vec_copy(s["r"], s["w"])
        lak.dense_gemv(s["V"].t(), s["h"], y=s["r"], alpha=-1.0, beta=1.0)
        lak.vec_dot(s["r"], s["r"], out=s["nrm"])
        return {"h": s["h"], "r": s["r"], "nrm": s["nrm"]}
    if kind == "chebyshev":
        rp, ci, v, _ = s["csr"]
        a, b = CHEB
        lak.csr_spmv(rp, ci, v, s["d"], y=s["q"])
        lak.vec_axpy_norm2(s["r2"], s["r"], s["q"], -1.0, out=s["nrm"])
        lak.vec_axpby(s["d2"], a, s["d"], b, s["r2"])
        lak.vec_axpy(s["u2"], s["u"], s["d2"], 1.0)
        return {"r": s["r2"], "nrm": s["nrm"], "d": s["d2"], "u": s["u2"]}
    if kind == "spmv":
        rp, ci, v, n = s["csr"]
        lak.csr_spmv(rp, ci, v, s["x"], y=s["y"], n_cols=n)
        return {"y": s["y"]}
    if kind in ("batch_gemv", "batch_spmv"):
        s["batch"].run()
        return {"y": s["y"]}
    if kind == "grad_dense":
        y = lak_autograd.gemv(s["A"], s["x"])
        loss = lak_autograd.dot(y, s["t"])
        dA, dx, dt = torch.autograd.grad(loss, (s["A"], s["x"], s["t"]))
        return {"loss": loss.detach(), "dA": dA, "dx": dx, "dt": dt}
    pattern = lak_autograd.CsrPattern(s["rp"], s["ci"], s["n"])
    y = lak_autograd.spmv(pattern, s["vals"], s["x"])
    dvals, dx = torch.autograd.grad(y, (s["vals"], s["x"]), s["dy"])
    return {"y": y.detach(), "dvals": dvals, "dx": dx}


# ---- what a pass cannot do without -------------------------------------------------

def _matrix_size(c):
    """(rows, entries) of a case's matrix (the power-law matrix: its mean)."""
    z = c["size"]
    if c["matrix"] == "powerlaw":
        return z, int(16 * z)
    if c["matrix"] == "elastic":
        return 3 * z ** 3, 9 * (3 * z - 2) ** 3
    return z ** 3, 7 * z ** 3 - 6 * z * z


def work(case):
    """Every input read once, every output written once."""
    kind, e = case["kind"], ESIZE[case["dtype"]]
    acc = 8 if e == 8 else 4
    if kind == "small":
        n, o = case["grid"] ** 2, case["order"]
        nnz = 5 * n - 4 * case["grid"]
        return {"bytes": 4 * n * e + nnz * (e + 4) + 4 * n + (o * o + 2 * o) * e + acc,
                "flops": 4 * n + 2 * nnz + 2 * o * o}
    if kind == "vectors":
        return {"bytes": 5 * case["n"] * e + 12, "flops": 6 * case["n"]}
    if kind == "lagged":
        return {"bytes": (2 * case["n"] + case["lag"]) * e + acc, "flops": 4 * case["n"]}
    if kind == "gemv":
        m, n = case["m"], case["n"]
        return {"bytes": (m * n + m + n) * e, "flops": 2 * m * n}
    if kind == "ortho":
        k, n = case["k"], case["n"]
        return {"bytes": (k * n + 2 * n + k + 1) * e, "flops": 4 * k * n + 2 * n}
    if kind == "chebyshev":
        m, nnz = _matrix_size({"matrix": "laplace", "size": case["grid"]})
        return {"bytes": nnz * (e + 4) + 4 * m + 6 * m * e + acc, "flops": 2 * nnz + 9 * m}
    if kind == "spmv":
        m, nnz = _matrix_size(case)
        return {"bytes": nnz * (e + 4) + 4 * m + 2 * m * e, "flops": 2 * nnz}
    if kind == "batch_gemv":
        mean = (4097 - 64) / math.log(4097 / 64)
        k = case["count"]
        return {"bytes": k * (mean * mean + 2 * mean) * e, "flops": 2 * k * mean * mean}
    if kind == "batch_spmv":
        rows = case["count"] * (200_001 - 1000) / math.log(200_001 / 1000)
        nnz = 34.5 * rows
        return {"bytes": nnz * (e + 4) + 4 * rows + 2 * rows * e, "flops": 2 * nnz}
    if kind == "grad_dense":
        m, n = case["m"], case["n"]
        return {"bytes": (2 * m * n + 2 * n + 2 * m + 1) * e, "flops": 5 * m * n + 4 * m}
    m, nnz = _matrix_size(case)
    return {"bytes": nnz * (2 * e + 4) + 4 * m + 4 * m * e, "flops": 5 * nnz}


# ---- the same results in 64 bits -----------------------------------------------------

def _spmv64(rp, ci, vals, x, m):
    rows = torch.arange(m, device=DEV).repeat_interleave((rp[1:] - rp[:-1]).long())
    out = torch.zeros(m, dtype=torch.float64, device=DEV)
    return out.index_add_(0, rows, vals.double() * x.double()[ci.long()])


def exact(case, seed):
    s = prepare(case, seed)
    kind = case["kind"]
    d = {k: v.detach().double() for k, v in s.items()
         if isinstance(v, torch.Tensor) and v.is_floating_point() and kind != "batch_gemv"}
    if kind == "small":
        rp, ci, v = s["csr"]
        x = d["y"] + 0.5 * d["z"]
        # the products are given the stored (rounded) update, as in run()
        xs = x.to(s["dtype"]).double()
        return {"x": x, "dot": (xs * d["y"]).sum().reshape(1),
                "q": _spmv64(rp, ci, v, xs, xs.numel()), "b": d["A"] @ d["v"]}
    if kind == "vectors":
        x = d["y"] + 0.5 * d["z"]
        xs = x.to(s["dtype"]).double()
        return {"x": x, "dot": (xs * d["y"]).sum().reshape(1),
                "cdot": (d["p"] * d["q"]).sum().reshape(1)}
    if kind == "lagged":
        return {"x": d["late"] - d["early"], "dot": (d["late"] * d["early"]).sum().reshape(1)}
    if kind == "gemv":
        return {"y": d["A"] @ d["x"]}
    if kind == "ortho":
        h = d["V"] @ d["w"]
        r = d["w"] - d["V"].t() @ h
        return {"h": h, "r": r, "nrm": (r * r).sum().reshape(1)}
    if kind == "chebyshev":
        rp, ci, v, _ = s["csr"]
        a, b = CHEB
        q = _spmv64(rp, ci, v, d["d"], d["d"].numel())
        r = d["r"] - q
        dn = a * d["d"] + b * r
        return {"r": r, "nrm": (r * r).sum().reshape(1), "d": dn, "u": d["u"] + dn}
    if kind == "spmv":
        rp, ci, v, _ = s["csr"]
        return {"y": _spmv64(rp, ci, v, s["x"], rp.numel() - 1)}
    if kind == "batch_gemv":
        out = torch.zeros(s["y"].numel(), dtype=torch.float64, device=DEV)
        base = s["y"].data_ptr()
        for A, x, y in zip(s["As"], s["xs"], s["ys"]):
            o = (y.data_ptr() - base) // y.element_size()
            torch.mv(A.double(), x.double(), out=out[o:o + y.numel()])
        return {"y": out}
    if kind == "batch_spmv":
        out = torch.zeros(s["y"].numel(), dtype=torch.float64, device=DEV)
        base = s["y"].data_ptr()
        for (rp, ci, v, m), x, y in zip(s["csrs"], s["xs"], s["ys"]):
            o = (y.data_ptr() - base) // y.element_size()
            out[o:o + m] = _spmv64(rp, ci, v, x, m)
        return {"y": out}
    if kind == "grad_dense":
        y = d["A"] @ d["x"]
        return {"loss": (y * d["t"]).sum(), "dA": torch.outer(d["t"], d["x"]),
                "dx": d["A"].t() @ d["t"], "dt": y}
    rp, ci, n = s["rp"], s["ci"], s["n"]
    rows = torch.arange(rp.numel() - 1, device=DEV).repeat_interleave((rp[1:] - rp[:-1]).long())
    cols = ci.long()
    dx = torch.zeros(n, dtype=torch.float64, device=DEV)
    dx.index_add_(0, cols, d["vals"] * d["dy"][rows])
    return {"y": _spmv64(rp, ci, d["vals"], d["x"], rp.numel() - 1),
            "dvals": d["dy"][rows] * d["x"][cols], "dx": dx}
