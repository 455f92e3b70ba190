"""The products, batches and solver calls that a program makes of this library, as timed cases.

Each case is a plain dict; ``prepare`` builds the matrix and the operands on the
GPU from a seed and creates the plan (batch, solver) that a program keeps, and
``run`` is one call of the public entry points.  Kinds:

* ``laplace2d``   5-point Laplacian on an nx x ny grid (constant coefficients)
* ``poisson3d``   7-point Poisson stencil with variable coefficients, nx x ny x nz
* ``stencil27``   27-point stencil (trilinear finite elements on a hexahedral grid)
* ``eigen``       symmetric matrix of an eigenproblem: diagonal, near bands kept with
                  p = 0.7, five scattered symmetric pairs per row
* ``powerlaw``    power-law row lengths (alpha = 2.2, at most 2000), uniform columns
* ``split``       the local/halo product of the Poisson matrix, the last tenth of the
                  columns arriving from pinned host memory
* ``batch``       many uneven power-law matrices in one launch
* ``cg``          conjugate gradients on the Poisson matrix
* ``lanczos``     Lanczos steps on the eigenproblem matrix

Plans are created with the library's defaults (the kernel is the plan's own
choice); ``fp32`` stores the values in FP32, ``k`` is the number of right-hand
sides and ``ld`` the leading dimension of their blocks.
"""
import math

import numpy as np
import torch

import paper_1101_0091_gb300 as spmv

DIM_LO, DIM_HI = 1e3, 2e5      # dimensions of a batch's members
ALPHA, LMAX = 2.2, 2000        # power-law row lengths
PAIRS, BAND_P = 5, 0.7         # eigenproblem matrix


def listed():
    return [
        # the smallest call: a 2D PDE on a 256 x 256 grid; launch and latency count
        {"name": "laplace2d_256", "kind": "laplace2d", "nx": 256, "ny": 256, "k": 1, "ld": 1, "fp32": False},
        # the largest: a 3D PDE on a 280^3 grid, one right-hand side; streams the matrix from HBM
        {"name": "poisson3d_280", "kind": "poisson3d", "nx": 280, "ny": 280, "nz": 280, "k": 1, "ld": 1, "fp32": False},
        # three components of a vector field advanced by one operator, odd grid and odd block
        {"name": "poisson3d_k3", "kind": "poisson3d", "nx": 131, "ny": 127, "nz": 129, "k": 3, "ld": 3, "fp32": False},
        # FP32-stored values with FP64 sums (a preconditioner's operator)
        {"name": "poisson3d_fp32", "kind": "poisson3d", "nx": 150, "ny": 151, "nz": 149, "k": 1, "ld": 1, "fp32": True},
        # finite elements: longer regular rows
        {"name": "stencil27", "kind": "stencil27", "nx": 101, "ny": 100, "nz": 99, "k": 1, "ld": 1, "fp32": False},
        # one product of an eigensolver: scattered gathers
        {"name": "eigen_2m", "kind": "eigen", "n": 2_000_003, "k": 1, "ld": 1, "fp32": False},
        # a block eigensolver's product on six vectors of an eight-column work block
        {"name": "eigen_k6", "kind": "eigen", "n": 600_011, "k": 6, "ld": 8, "fp32": False},
        # one matrix with very uneven rows (graphs, circuits), the largest of the uneven batch
        {"name": "powerlaw_200k", "kind": "powerlaw", "n": 200_000, "k": 1, "ld": 1, "fp32": False},
        # domain decomposition: the halo of B arrives from the host during the local product
        {"name": "split_150", "kind": "split", "nx": 150, "ny": 149, "nz": 151, "k": 1, "ld": 1, "fp32": False},
        # the uneven batch: 512 small systems, four right-hand sides each
        {"name": "batch_512_k4", "kind": "batch", "count": 512, "k": 4, "ld": 4},
        # a linear solve's iterations (a fixed number, as inside an outer iteration)
        {"name": "cg_128", "kind": "cg", "nx": 128, "ny": 128, "nz": 128, "k": 1, "steps": 40},
        # a block Lanczos run for the extreme eigenvalues
        {"name": "lanczos_k4", "kind": "lanczos", "n": 500_009, "k": 4, "steps": 20},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _grid3(rng, lo, hi):
    """Edges of a 3D grid of lo .. hi points in all, near-cubic, ragged."""
    n = _log_int(rng, lo, hi)
    e = n ** (1.0 / 3.0)
    nx = max(2, int(round(e * rng.uniform(0.8, 1.25))))
    ny = max(2, int(round(e * rng.uniform(0.8, 1.25))))
    return {"nx": nx, "ny": ny, "nz": max(2, n // (nx * ny))}


def draw(rng):
    kind = rng.choice(["laplace2d", "poisson3d", "poisson3d", "stencil27", "eigen", "eigen", "powerlaw", "split",
                       "batch", "cg", "lanczos"])
    k = rng.choice([1, 1, 1, 2, 3, 4, 5, 6, 7, 8, 12, 13, 16])
    ld = k + (rng.choice([0, 0, 1, 2, 3]) if k > 1 else 0)
    block = {"k": k, "ld": ld, "fp32": rng.random() < 0.25}
    if kind == "laplace2d":
        nx = _log_int(rng, 30, 1500)
        return {"kind": kind, "nx": nx, "ny": _log_int(rng, 30, 1500), **block}
    if kind in ("poisson3d", "stencil27"):
        return {"kind": kind, **_grid3(rng, 2e4, (8e6 if kind == "poisson3d" else 1.2e6) / math.sqrt(k)), **block}
    if kind == "eigen":
        return {"kind": kind, "n": _log_int(rng, 2e4, 2.5e6 / math.sqrt(k)), **block}
    if kind == "powerlaw":
        return {"kind": kind, "n": _log_int(rng, DIM_LO, DIM_HI), **block}
    if kind == "split":
        return {"kind": kind, **_grid3(rng, 2e4, 4e6), "k": 1, "ld": 1, "fp32": rng.random() < 0.25}
    if kind == "batch":
        kb = rng.choice([1, 2, 3, 4, 4, 4, 8, 16])
        return {"kind": kind, "count": _log_int(rng, 16, 128 if kb > 4 else 400), "k": kb, "ld": kb}
    if kind == "cg":
        return {"kind": kind, **_grid3(rng, 2e4, 2.5e6 / k), "k": k, "steps": rng.randint(10, 40)}
    return {"kind": kind, "n": _log_int(rng, 2e4, 1e6 / math.sqrt(k)), "k": k, "steps": rng.randint(8, 24)}


# ------------------------------------------------------------------ inputs
def _gen(seed, stream):
    g = torch.Generator(device="cuda")
    g.manual_seed(1_000_003 * int(seed) + stream)
    return g


def _uniform(shape, g, lo=-1.0, hi=1.0):
    return torch.rand(shape, generator=g, device="cuda", dtype=torch.float64) * (hi - lo) + lo


def _compact(cols, vals, keep):
    """Row-major compaction of an n x m table of entries into CRS."""
    rp = torch.zeros(keep.shape[0] + 1, dtype=torch.int64, device="cuda")
    rp[1:] = torch.cumsum(keep.sum(1), 0)
    return rp.to(torch.int32), cols[keep], vals[keep]


def _stencil(nx, ny, nz, kind, g):
    n = nx * ny * nz
    i = torch.arange(n, device="cuda", dtype=torch.int32)
    x, y, z = i % nx, (i // nx) % ny, i // (nx * ny)
    if kind == "stencil27":
        offs = [(a, b, c) for c in (-1, 0, 1) for b in (-1, 0, 1) for a in (-1, 0, 1)]
    elif kind == "laplace2d":
        offs = [(0, -1, 0), (-1, 0, 0), (0, 0, 0), (1, 0, 0), (0, 1, 0)]
    else:
        offs = [(0, 0, -1), (0, -1, 0), (-1, 0, 0), (0, 0, 0), (1, 0, 0), (0, 1, 0), (0, 0, 1)]
    m = len(offs)
    keep = torch.empty((n, m), dtype=torch.bool, device="cuda")
    cols = torch.empty((n, m), dtype=torch.int32, device="cuda")
    for s, (a, b, c) in enumerate(offs):
        keep[:, s] = (x + a >= 0) & (x + a < nx) & (y + b >= 0) & (y + b < ny) & (z + c >= 0) & (z + c < nz)
        cols[:, s] = i + (a + nx * (b + ny * c))
    del x, y, z
    mid = offs.index((0, 0, 0))
    if kind == "laplace2d":
        vals = torch.full((n, m), -1.0, dtype=torch.float64, device="cuda")
        vals[:, mid] = 4.0
        return _compact(cols, vals, keep)
    vals = torch.zeros((n, m), dtype=torch.float64, device="cuda")
    for s in range(mid + 1, m):   # one coefficient per edge, the same seen from both of its ends
        w = -(1.0 + torch.rand(n, generator=g, device="cuda", dtype=torch.float64))
        vals[:, s] = w
        o = offs[s][0] + nx * (offs[s][1] + ny * offs[s][2])
        vals[o:, m - 1 - s] = w[:n - o]
    vals[~keep] = 0.0
    vals[:, mid] = vals.abs().sum(1) + 1e-3
    return _compact(cols, vals, keep)


def _from_coo(n, rows, cols, vals):
    order = torch.argsort(rows * n + cols, stable=True)
    rp = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    rp[1:] = torch.cumsum(torch.bincount(rows, minlength=n), 0)
    return rp.to(torch.int32), cols[order].to(torch.int32), vals[order]


def _eigen(n, g):
    i = torch.arange(n, device="cuda", dtype=torch.int64)
    rows, cols, vals = [i], [i], [torch.randn(n, generator=g, device="cuda", dtype=torch.float64)]
    window = max(4, min(1 << 20, n // 3))

    def mirrored(r, c):
        v = _uniform(r.shape[0], g)
        rows.extend([r, c])
        cols.extend([c, r])
        vals.extend([v, v])

    for d in (1, 2):
        r = i[:n - d][torch.rand(n - d, generator=g, device="cuda") < BAND_P]
        mirrored(r, r + d)
    for _ in range(PAIRS):
        d = torch.randint(3, window + 1, (n,), generator=g, device="cuda")
        d = torch.where(torch.rand(n, generator=g, device="cuda") < 0.5, d, -d)
        c = i + d
        c = torch.where((c < 0) | (c >= n), i - d, c)
        mirrored(i, c)
    return _from_coo(n, torch.cat(rows), torch.cat(cols), torch.cat(vals))


def _powerlaw_lengths(n, cap, g):
    """Lengths with P(L) ~ L^-alpha on 1 .. cap (cap: one value, or one per row)."""
    p = torch.cumsum(torch.arange(1, LMAX + 1, dtype=torch.float64, device="cuda") ** -ALPHA, 0)
    u = torch.rand(n, generator=g, device="cuda", dtype=torch.float64) * p[torch.as_tensor(cap, device="cuda") - 1]
    return torch.searchsorted(p, u).clamp_(max=LMAX - 1) + 1


def _powerlaw(n, g):
    lens = _powerlaw_lengths(n, min(LMAX, n), g)
    rows = torch.repeat_interleave(torch.arange(n, device="cuda"), lens)
    nnz = rows.shape[0]
    cols = (torch.rand(nnz, generator=g, device="cuda", dtype=torch.float64) * n).long().clamp_(max=n - 1)
    return _from_coo(n, rows, cols, _uniform(nnz, g))


def _batch_dims(count):
    """Member dimensions, spread evenly over the logarithm, in a mixed order."""
    u = (np.random.RandomState(count).permutation(count) + 0.5) / count
    return np.round(DIM_LO * (DIM_HI / DIM_LO) ** u).astype(np.int64)


def _batch_members(count, seed):
    """Member dimensions and the CRS arrays of all members, one after another (columns are each member's own)."""
    g = _gen(seed, 1)
    dims = torch.from_numpy(_batch_dims(count)).cuda()
    dim_of_row = torch.repeat_interleave(dims, dims)
    lens = _powerlaw_lengths(dim_of_row.shape[0], dim_of_row.clamp(max=LMAX), g)
    rows = torch.repeat_interleave(torch.arange(lens.shape[0], device="cuda"), lens)
    nnz = rows.shape[0]
    d = dim_of_row[rows]
    cols = torch.minimum((torch.rand(nnz, generator=g, device="cuda", dtype=torch.float64) * d).long(), d - 1)
    order = torch.argsort(rows * int(DIM_HI + 1) + cols, stable=True)
    rp = torch.zeros(lens.shape[0] + 1, dtype=torch.int64, device="cuda")
    rp[1:] = torch.cumsum(lens, 0)
    return dims, rp, rows, cols[order], _uniform(nnz, g)


def _matrix(case, seed):
    """(n, row_ptr, col, val) on the GPU."""
    g = _gen(seed, 1)
    kind = case["kind"]
    if kind in ("eigen", "lanczos"):
        return (case["n"], *_eigen(case["n"], g))
    if kind == "powerlaw":
        return (case["n"], *_powerlaw(case["n"], g))
    nz = case.get("nz", 1)
    kind = "poisson3d" if kind in ("split", "cg") else kind
    return (case["nx"] * case["ny"] * nz, *_stencil(case["nx"], case["ny"], nz, kind, g))


def _rhs(n, case, seed):
    """Block of right-hand sides, U[-1, 1): n x ld, the first k columns used (k = ld = 1: a vector)."""
    k, ld = case["k"], case.get("ld", case["k"])
    g = _gen(seed, 2)
    return _uniform(n, g) if k == ld == 1 else _uniform((n, ld), g)


def prepare(case, seed):
    kind, k = case["kind"], case["k"]
    if kind == "batch":
        dims, rp, _, cols, vals = _batch_members(case["count"], seed)
        ends = torch.cumsum(dims, 0).tolist()
        rp, cols, vals = rp.cpu().numpy(), cols.to(torch.int32).cpu().numpy(), vals.cpu().numpy()
        plans, spans, r0 = [], [], 0
        for r1 in ends:
            p = rp[r0:r1 + 1]
            plans.append(spmv.Plan(r1 - r0, r1 - r0, (p - p[0]).astype(np.int32), cols[p[0]:p[-1]], vals[p[0]:p[-1]]))
            spans.append((r0, r1))
            r0 = r1
        B = _uniform((r0, k), _gen(seed, 2))
        C = torch.zeros((r0, k), dtype=torch.float64, device="cuda")
        batch = spmv.Batch(plans, k)
        batch.set_io([B[a:b] for a, b in spans], [C[a:b] for a, b in spans])
        return {"kind": kind, "batch": batch, "B": B, "C": C}
    n, rp, ci, va = _matrix(case, seed)
    rp, ci, va = rp.cpu().numpy(), ci.cpu().numpy(), va.cpu().numpy()
    if kind == "split":
        h = n - n // 10
        plan = spmv.Plan(n, n, rp, ci, va, val_fp32=case["fp32"], halo_begin=h)
        B = _rhs(n, case, seed)
        halo = B[h:].cpu().pin_memory()
        return {"kind": kind, "plan": plan, "B": B, "halo": halo, "C": torch.zeros_like(B),
                "copy": torch.cuda.Stream()}
    plan = spmv.Plan(n, n, rp, ci, va, val_fp32=case.get("fp32", False))
    if kind in ("cg", "lanczos"):
        B = _uniform((n, k), _gen(seed, 2))
        return {"kind": kind, "solver": spmv.Solver(plan, k), "B": B, "X": torch.zeros_like(B),
                "steps": case["steps"]}
    B = _rhs(n, case, seed)
    return {"kind": kind, "plan": plan, "B": B, "C": torch.zeros_like(B), "k": k}


def run(state):
    kind = state["kind"]
    if kind == "batch":
        state["batch"].apply()
        return state["C"]
    if kind == "split":
        state["plan"].apply_split(state["B"], state["halo"], state["C"], copy_stream=state["copy"])
        return {"C": state["C"], "B": state["B"]}
    if kind == "cg":
        state["X"].zero_()
        iterations, rr, _ = state["solver"].cg(state["B"], state["X"], max_iter=state["steps"], rtol=1e-12)
        return {"X": state["X"], "iterations": iterations, "rr": rr}
    if kind == "lanczos":
        alpha, beta = state["solver"].lanczos(state["B"], state["steps"])
        return {"alpha": alpha, "beta": beta}
    if state["B"].dim() == 1:
        state["plan"].apply(state["B"], state["C"])
    else:
        state["plan"].apply_block(state["B"], state["C"], state["k"])
    return state["C"]


# ------------------------------------------------------------------ work and 64-bit values
def _mean_length():
    w = np.arange(1, LMAX + 1, dtype=np.float64) ** -ALPHA
    return float((w * np.arange(1, LMAX + 1)).sum() / w.sum())


def _size(case):
    """(rows, nonzeros) of a case's matrix; expected values where they depend on the seed."""
    kind = case["kind"]
    if kind == "batch":
        n = int(_batch_dims(case["count"]).sum())
        return n, n * _mean_length()
    if kind == "powerlaw":
        return case["n"], case["n"] * _mean_length()
    if kind in ("eigen", "lanczos"):
        return case["n"], case["n"] * (1 + 4 * BAND_P + 2 * PAIRS)
    nx, ny, nz = case["nx"], case["ny"], case.get("nz", 1)
    n = nx * ny * nz
    if kind == "stencil27":
        return n, (3 * nx - 2) * (3 * ny - 2) * (3 * nz - 2)
    return n, n + 2 * ((nx - 1) * ny * nz + nx * (ny - 1) * nz + nx * ny * (nz - 1))


def work(case):
    """One pass: the matrix, B and C once per product, two operations per nonzero and right-hand side; the solvers'
    vector updates read and write each of their vectors once per step."""
    n, nnz = _size(case)
    k = case["k"]
    product = nnz * ((4 if case.get("fp32") else 8) + 4) + 4 * (n + 1) + 16 * k * n
    flops = 2 * k * nnz
    if case["kind"] == "cg":          # X, R, P read and written, Q written by the product and read
        return {"bytes": case["steps"] * (product + 8 * k * n * 5), "flops": case["steps"] * (flops + 10 * k * n)}
    if case["kind"] == "lanczos":     # the previous vector read, the new one read and written
        return {"bytes": case["steps"] * (product + 8 * k * n * 3), "flops": case["steps"] * (flops + 9 * k * n)}
    return {"bytes": product, "flops": flops}


def _product(rows, ci, va, B, n):
    """A * B (n x k) by a sum over the entries of each row, 64 bits."""
    C = torch.zeros((n, B.shape[1]), dtype=torch.float64, device="cuda")
    step = max(1, (1 << 28) // B.shape[1])
    for a in range(0, rows.shape[0], step):
        C.index_add_(0, rows[a:a + step], va[a:a + step, None] * B[ci[a:a + step].long()])
    return C


def exact(case, seed):
    kind, k = case["kind"], case["k"]
    if kind == "batch":
        dims, _, rows, cols, vals = _batch_members(case["count"], seed)
        first = torch.cumsum(dims, 0) - dims
        n = int(dims.sum())
        B = _uniform((n, k), _gen(seed, 2))
        return _product(rows, cols + torch.repeat_interleave(first, dims)[rows], vals, B, n)
    n, rp, ci, va = _matrix(case, seed)
    rows = torch.repeat_interleave(torch.arange(n, device="cuda"), (rp[1:] - rp[:-1]).long())
    if case.get("fp32"):   # the option stores the rounded values
        va = va.float().double()
    if kind in ("cg", "lanczos"):
        B = _uniform((n, k), _gen(seed, 2))
        return (_exact_cg if kind == "cg" else _exact_lanczos)(lambda V: _product(rows, ci, va, V, n), B,
                                                               case["steps"])
    B = _rhs(n, case, seed)
    if B.dim() == 1:
        C = _product(rows, ci, va, B[:, None], n)[:, 0]
        return {"C": C, "B": B} if kind == "split" else C
    C = torch.zeros_like(B)
    C[:, :k] = _product(rows, ci, va, B[:, :k], n)
    return C


def _exact_cg(apply, B, steps):
    X, R, P = torch.zeros_like(B), B.clone(), B.clone()
    rr = (R * R).sum(0)
    for _ in range(steps):
        Q = apply(P)
        alpha = rr / (P * Q).sum(0)
        X += alpha * P
        R -= alpha * Q
        new = (R * R).sum(0)
        P = R + (new / rr) * P
        rr = new
    return {"X": X, "iterations": None, "rr": rr.cpu().numpy()}


def _exact_lanczos(apply, B, steps):
    v = B / B.norm(dim=0)
    prev, beta, al, be = torch.zeros_like(v), torch.zeros(B.shape[1], dtype=torch.float64, device="cuda"), [], []
    for _ in range(steps):
        w = apply(v) - beta * prev
        a = (w * v).sum(0)
        w -= a * v
        beta = w.norm(dim=0)
        al.append(a)
        be.append(beta)
        prev, v = v, w / beta
    return {"alpha": torch.stack(al).cpu().numpy(), "beta": torch.stack(be).cpu().numpy()}
