"""Performance cases of the sparse product library: what a program that uses
it has it do, through the public entry points of the Python binding.

The inputs are built on the GPU from a seed: the multigrid operators (stencil
matrices with a varying coefficient, smoothed-aggregation prolongators),
R-MAT graphs (edge weights in [0.5, 1.5)) and uniform random rows of the
library's own tests and benchmark.  A case keeps its sizes from seed to seed.

  listed()             the fixed cases
  draw(rng)            one more case of the same ranges
  prepare(case, seed)  what a program holds before the call
  run(state)           one pass, and its outputs
  work(case)           bytes and operations a pass cannot do without
  exact(case, seed)    the outputs in 64 bits, by plain torch
"""
import math
import random

import torch

import paper_1804_00695_gb300 as sg

DEV = "cuda"
DTYPES = {"f32": torch.float32, "f64": torch.float64}


# ------------------------------------------------------------------- cases
def listed():
    return [
        # A*A of a 5-point Laplacian on a 64 x 64 grid: a small product whose
        # time is launches and the host's waits, as in the inner loops of a
        # solver's setup on its coarse levels
        {"name": "square_2d_64", "kind": "square", "family": "laplace2d_5pt", "n": 64, "dtype": "f64"},
        # the Galerkin triple product R*(A*P) of a multigrid setup: a middle
        # level on an odd grid, and the finest level of the benchmark
        {"name": "galerkin_45", "kind": "galerkin", "family": "brick3d_27pt", "n": 45, "dtype": "f64"},
        {"name": "galerkin_128", "kind": "galerkin", "family": "brick3d_27pt", "n": 128, "dtype": "f64"},
        # the numeric phase alone, the patterns of an earlier symbolic phase
        # kept: a time-stepping or nonlinear solve whose coefficients change
        {"name": "renumeric_100", "kind": "renumeric", "family": "brick3d_27pt", "n": 100, "dtype": "f32"},
        # the triple product of 3D elasticity: 81 entries a row, blocks of 3
        {"name": "elasticity_32", "kind": "galerkin", "family": "elasticity3d_81", "n": 32, "dtype": "f64"},
        # elasticity operator times a random right-hand side of about 64
        # entries a row (the density experiment): long rows, few collisions
        {"name": "density_24_64", "kind": "density", "family": "elasticity3d_81", "n": 24, "delta": 64,
         "dtype": "f64"},
        # A*A of a power-law graph (two-hop neighbours): small and large
        {"name": "rmat_13", "kind": "rmat", "scale": 13, "edges": 16, "dtype": "f32"},
        {"name": "rmat_17", "kind": "rmat", "scale": 17, "edges": 16, "dtype": "f32"},
        # 64 independent products in one call, ragged sizes
        {"name": "batched_64", "kind": "batched", "count": 64, "lo": 1024, "hi": 65536, "dtype": "f32"},
        # forward and backward of a differentiable product
        {"name": "autograd_20001", "kind": "autograd", "n": 20001, "dtype": "f32"},
        # triangles of a power-law graph by the masked product
        {"name": "triangles_18", "kind": "triangles", "scale": 18, "edges": 16},
        # operands and result in host memory, streamed through a device budget
        {"name": "chunked_96", "kind": "chunked", "family": "brick3d_27pt", "n": 96, "budget_mb": 256, "dtype": "f64"},
    ]


#: largest grid of a drawn multigrid product, by family
MOST_N = {"laplace2d_5pt": 1200, "bigstar2d_13pt": 1000, "laplace3d_7pt": 150, "brick3d_27pt": 120,
          "elasticity3d_81": 32}


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["square", "galerkin", "galerkin", "renumeric", "density", "rmat", "batched", "autograd",
                       "triangles", "chunked"])
    dtype = rng.choice(["f32", "f64", "f64"])
    if kind in ("square", "galerkin", "renumeric"):
        family = rng.choice(sorted(MOST_N))
        most = MOST_N[family] if kind != "square" else MOST_N[family] * 2 // 3
        return {"kind": kind, "family": family, "n": _log_int(rng, 12 if "3d" in family else 30, most), "dtype": dtype}
    if kind == "density":
        return {"kind": kind, "family": rng.choice(["elasticity3d_81", "brick3d_27pt"]), "n": rng.randint(10, 24),
                "delta": _log_int(rng, 1, 200), "dtype": dtype}
    if kind == "rmat":
        return {"kind": kind, "scale": rng.randint(10, 16), "edges": rng.randint(4, 16), "dtype": dtype}
    if kind == "batched":
        return {"kind": kind, "count": _log_int(rng, 3, 200), "lo": _log_int(rng, 64, 2048),
                "hi": _log_int(rng, 4096, 40000), "dtype": dtype}
    if kind == "autograd":
        return {"kind": kind, "n": _log_int(rng, 500, 100000), "dtype": dtype}
    if kind == "triangles":
        return {"kind": kind, "scale": rng.randint(10, 18), "edges": rng.randint(4, 15)}
    return {"kind": kind, "family": rng.choice(["brick3d_27pt", "laplace3d_7pt"]), "n": rng.randint(30, 95),
            "budget_mb": rng.choice([256, 384, 512]), "dtype": dtype}


# ------------------------------------------------------------------- inputs
def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(seed)


def _offsets(rows, nrows):
    rp = torch.zeros(nrows + 1, dtype=torch.int64, device=DEV)
    torch.cumsum(torch.bincount(rows, minlength=nrows), 0, out=rp[1:])
    return rp


def _csr(rows, cols, vals, nrows, ncols):
    """Entries already in row-major order, as the library's CSR."""
    return sg.Csr(nrows, ncols, _offsets(rows, nrows), cols.to(torch.int32), vals)


def _box(d):
    return [tuple((k // 3 ** j) % 3 - 1 for j in range(d)) for k in range(3 ** d)]


STENCILS = {
    "laplace2d_5pt": (2, [(0, 0), (1, 0), (-1, 0), (0, 1), (0, -1)], 1),
    "bigstar2d_13pt": (2, [(0, 0), (1, 0), (-1, 0), (0, 1), (0, -1), (1, 1), (1, -1), (-1, 1), (-1, -1), (2, 0),
                           (-2, 0), (0, 2), (0, -2)], 1),
    "laplace3d_7pt": (3, [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1)], 1),
    "brick3d_27pt": (3, _box(3), 1),
    "elasticity3d_81": (3, _box(3), 3),
}


def _stencil(family, n, dtype, gen):
    """Operator on an n^d grid with a varying coefficient (b unknowns a point,
    coupled by full b x b blocks), and its scalar pattern (rows, columns)."""
    d, offs, b = STENCILS[family]
    lin = sorted((sum(o[k] * n ** k for k in range(d)), o) for o in offs)
    N = n ** d
    row = torch.arange(N, device=DEV)
    ok = torch.ones((N, len(lin)), dtype=torch.bool, device=DEV)
    for k in range(d):
        x = (row // n ** k) % n
        o = torch.tensor([v[1][k] for v in lin], device=DEV)
        y = x[:, None] + o[None, :]
        ok &= (y >= 0) & (y < n)
    disp = torch.tensor([v[0] for v in lin], device=DEV)
    col = row[:, None] + disp[None, :]
    srow, scol = row[:, None].expand_as(col)[ok], col[ok]
    if b == 1:
        rows, cols = srow, scol
    else:
        r = torch.arange(b, device=DEV)
        full = (N, b, len(lin), b)
        keep = ok[:, None, :, None].expand(full)
        rows = (row[:, None] * b + r)[:, :, None, None].expand(full)[keep]
        cols = (col[:, None, :, None] * b + r).expand(full)[keep]
    u = torch.rand(rows.numel(), dtype=dtype, device=DEV, generator=gen) + 0.5
    vals = torch.where(rows == cols, u * len(lin), -u)
    return _csr(rows, cols, vals, N * b, N * b), srow, scol


def _prolongator(family, n, srow, scol, dtype, gen):
    """Smoothed aggregation over 3 points a dimension: the pattern of
    A * P_tent, weights falling off with the distance."""
    d, _, b = STENCILS[family]
    nc = (n + 2) // 3
    agg = torch.zeros_like(scol)
    for k in range(d):
        agg += ((scol // n ** k) % n) // 3 * nc ** k
    key = torch.unique(srow * nc ** d + agg)
    rows, cols = key // nc ** d, key % nc ** d
    if b > 1:
        r = torch.arange(b, device=DEV)
        key = ((rows[:, None, None] * b + r[None, :, None]) * (nc ** d * b) + cols[:, None, None] * b + r).reshape(-1)
        key = torch.sort(key).values
        rows, cols = key // (nc ** d * b), key % (nc ** d * b)
    vals = torch.rand(rows.numel(), dtype=dtype, device=DEV, generator=gen) * 0.3 + 0.02
    return _csr(rows, cols, vals, n ** d * b, nc ** d * b)


def _row_ids(m):
    return torch.repeat_interleave(torch.arange(m.nrows, device=DEV), m.row_ptr[1:] - m.row_ptr[:-1])


def _transpose(m):
    order = torch.argsort(m.col, stable=True)
    return _csr(m.col[order].to(torch.int64), _row_ids(m)[order], m.val[order], m.ncols, m.nrows)


def _multigrid(case, seed):
    gen, dtype = _gen(seed), DTYPES[case["dtype"]]
    A, srow, scol = _stencil(case["family"], case["n"], dtype, gen)
    P = _prolongator(case["family"], case["n"], srow, scol, dtype, gen)
    return A, P, _transpose(P)


def _random_rows(nrows, ncols, lo, hi, dtype, pattern, gen, shift=0):
    """lo..hi uniform random columns a row (repeats dropped) from the seed
    `pattern`, moved on by `shift` columns (the product keeps its size when
    the right operand's columns move); N(0,1) values from gen."""
    pat = _gen(pattern)
    length = torch.randint(lo, hi + 1, (nrows,), device=DEV, generator=pat)
    cand = (torch.randint(0, ncols, (nrows, hi), device=DEV, generator=pat) + shift) % ncols
    take = torch.arange(hi, device=DEV)[None, :] < length[:, None]
    key = torch.unique((torch.arange(nrows, device=DEV)[:, None] * ncols + cand)[take])
    vals = torch.randn(key.numel(), dtype=dtype, device=DEV, generator=gen)
    return _csr(key // ncols, key % ncols, vals, nrows, ncols)


def _rmat(scale, edges, pattern):
    """Pattern of a symmetrised R-MAT graph (.57, .19, .19, .05), no loops."""
    gen, n = _gen(pattern), 1 << scale
    m = edges * n
    r = torch.zeros(m, dtype=torch.int64, device=DEV)
    c = torch.zeros(m, dtype=torch.int64, device=DEV)
    for _ in range(scale):
        u = torch.rand(m, device=DEV, generator=gen)
        r = 2 * r + (u >= 0.76)
        c = 2 * c + (((u >= 0.57) & (u < 0.76)) | (u >= 0.95))
    r, c = r[r != c], c[r != c]
    key = torch.unique(torch.cat([r * n + c, c * n + r]))
    return _csr(key // n, key % n, None, n, n)


def _batch(case, seed):
    gen, dtype = _gen(seed), DTYPES[case["dtype"]]
    sizes = random.Random(case["count"])
    out = []
    for i in range(case["count"]):
        n = _log_int(sizes, case["lo"], case["hi"])
        out.append((_random_rows(n, n, 4, 32, dtype, 2 * i, gen),
                    _random_rows(n, n, 4, 32, dtype, 2 * i + 1, gen, shift=seed)))
    return out


def _operands(case, seed):
    """The products of a pass: a list of (A, B) on the device; None in the
    place of a B that is the product before it."""
    kind = case["kind"]
    if kind in ("square", "chunked"):
        A = _stencil(case["family"], case["n"], DTYPES[case["dtype"]], _gen(seed))[0]
        return [(A, sg.Csr(A.nrows, A.ncols, A.row_ptr.clone(), A.col.clone(), A.val.clone()))]
    if kind in ("galerkin", "renumeric"):
        A, P, R = _multigrid(case, seed)
        return [(A, P), (R, None)]
    if kind == "density":
        gen, dtype = _gen(seed), DTYPES[case["dtype"]]
        A = _stencil(case["family"], case["n"], dtype, gen)[0]
        return [(A, _random_rows(A.ncols, A.ncols, case["delta"], case["delta"], dtype, 1, gen, shift=seed))]
    if kind == "rmat":
        A = _rmat(case["scale"], case["edges"], 1)
        A.val = torch.rand(A.nnz, dtype=DTYPES[case["dtype"]], device=DEV, generator=_gen(seed)) + 0.5
        return [(A, A)]
    if kind == "batched":
        return _batch(case, seed)
    gen, dtype = _gen(seed), DTYPES[case["dtype"]]   # autograd
    n = case["n"]
    return [(_random_rows(n, n, 4, 32, dtype, 1, gen), _random_rows(n, n, 4, 32, dtype, 2, gen, shift=seed))]


def _host(m):
    return sg.HostCsr(m.nrows, m.ncols, *(t.cpu().pin_memory() for t in (m.row_ptr, m.col, m.val)))


def _upstream(nnz, dtype, seed):
    return torch.randn(nnz, dtype=dtype, device=DEV, generator=_gen(seed + 7919))


# -------------------------------------------------------------------- state
def prepare(case, seed):
    kind = case["kind"]
    state = {"kind": kind, "h": sg.Handle()}
    if kind == "triangles":
        state["G"] = _rmat(case["scale"], case["edges"], seed)
        return state
    ops = _operands(case, seed)
    if kind == "batched":
        state["batch"] = sg.Batch(state["h"], [a for a, _ in ops], [b for _, b in ops])
    elif kind in ("galerkin", "renumeric"):
        (state["A"], state["P"]), (state["R"], _) = ops
        if kind == "renumeric":
            # a handle for each of the two products keeps its pattern
            state["h2"] = sg.Handle()
            state["AP"] = state["h"].spgemm(state["A"], state["P"])
            state["RAP"] = state["h2"].spgemm(state["R"], state["AP"])
    elif kind == "chunked":
        state["A"], state["B"] = (_host(m) for m in ops[0])
        state["budget"] = case["budget_mb"] << 20
    else:
        state["A"], state["B"] = ops[0]
        if kind == "autograd":
            _, nnz = state["h"].symbolic(state["A"], state["B"])
            state["dC"] = _upstream(nnz, state["A"].val.dtype, seed)
            state["A"].val.requires_grad_(True)
            state["B"].val.requires_grad_(True)
    return state


def _out(m):
    return [m.row_ptr, m.col, m.val]


def run(state):
    kind, h = state["kind"], state["h"]
    if kind == "galerkin":
        AP = h.spgemm(state["A"], state["P"])
        return _out(AP) + _out(h.spgemm(state["R"], AP))
    if kind == "renumeric":
        h.numeric_into(state["A"], state["P"], state["AP"])
        state["h2"].numeric_into(state["R"], state["AP"], state["RAP"])
        return _out(state["AP"]) + _out(state["RAP"])
    if kind == "batched":
        return _out(state["batch"].run())
    if kind == "autograd":
        A, B = state["A"], state["B"]
        C = sg.spgemm_autograd(A, B, h)
        return [C.row_ptr, C.col, C.val.detach(), *torch.autograd.grad(C.val, (A.val, B.val), state["dC"])]
    if kind == "triangles":
        return h.triangles(state["G"])
    if kind == "chunked":
        return _out(h.chunked(state["A"], state["B"], state["budget"]))
    return _out(h.spgemm(state["A"], state["B"]))


# --------------------------------------------------------------------- work
def _lengths(m):
    return m.row_ptr[1:] - m.row_ptr[:-1]


def _products(A, B):
    return int(_lengths(B)[A.col.to(torch.int64)].sum())


def work(case):
    """Operands read once, results written once; a multiplication and an
    addition for each product a_ik * b_kj."""
    def size(m, nnz=None):   # offsets, columns and values of a matrix
        return 8 * (m.nrows + 1) + (m.nnz if nnz is None else nnz) * (4 + m.val.element_size())

    if case["kind"] == "triangles":
        # the pattern in, the count out; a triangle test for every pair of
        # entries L_ik, L_kj of the degree-ordered lower triangle
        G = _rmat(case["scale"], case["edges"], 0)
        deg, row, col = _lengths(G), _row_ids(G), G.col.to(torch.int64)
        order = deg * G.nrows + torch.arange(G.nrows, device=DEV)
        low = order[col] < order[row]
        lower = torch.bincount(row[low], minlength=G.nrows)
        return {"bytes": 8 * (G.nrows + 1) + 4 * G.nnz + 8, "flops": 2 * int(lower[col[low]].sum())}
    h, bytes_, flops, C = sg.Handle(), 0, 0, None
    for A, B in _operands(case, 0):
        B = C if B is None else B
        rp, nnz = h.symbolic(A, B)
        p = _products(A, B)
        if case["kind"] == "renumeric":
            bytes_ += 8 * (A.nrows + 1)   # the offsets of C are read
        bytes_ += size(A) + (0 if B is A else size(B)) + 8 * (A.nrows + 1) + nnz * (4 + A.val.element_size())
        flops += 2 * p
        if case["kind"] == "autograd":
            # dC and the operands read again, both gradients written
            bytes_ += nnz * (4 + A.val.element_size()) + size(A) + size(B) + (A.nnz + B.nnz) * A.val.element_size()
            flops += 4 * p
        if case["kind"] in ("galerkin", "renumeric"):
            C = h.numeric(A, B, rp, nnz)
    return {"bytes": bytes_, "flops": flops}


# -------------------------------------------------------------------- exact
MOST_PRODUCTS = 1 << 27   # products expanded at a time


def _expand(A, B, r0, r1):
    """Every product of rows r0..r1 of A*B: entry of A, entry of B, and
    row * ncols + column."""
    p0, p1 = int(A.row_ptr[r0]), int(A.row_ptr[r1])
    k = A.col[p0:p1].to(torch.int64)
    cnt = _lengths(B)[k]
    ea = torch.repeat_interleave(torch.arange(p0, p1, device=DEV), cnt)
    first = torch.cumsum(cnt, 0) - cnt
    eb = torch.arange(ea.numel(), device=DEV) - torch.repeat_interleave(first - B.row_ptr[k], cnt)
    row = torch.repeat_interleave(torch.arange(r0, r1, device=DEV), _lengths(A)[r0:r1])
    key = torch.repeat_interleave(row, cnt) * B.ncols + B.col[eb].to(torch.int64)
    return ea, eb, key


def _row_blocks(A, B):
    cum = torch.cumsum(_lengths(B)[A.col.to(torch.int64)], 0)
    per_row = torch.cat([cum.new_zeros(1), cum])[A.row_ptr].cpu()
    r0 = 0
    while r0 < A.nrows:
        r1 = int(torch.searchsorted(per_row, per_row[r0] + MOST_PRODUCTS, right=True)) - 1
        r1 = min(A.nrows, max(r1, r0 + 1))
        yield r0, r1
        r0 = r1


def _exact_product(A, B):
    """A*B with 64-bit values, by expanding and sorting all products."""
    av, bv = A.val.detach().double(), B.val.detach().double()
    lens, cols, vals = [], [], []
    for r0, r1 in _row_blocks(A, B):
        ea, eb, key = _expand(A, B, r0, r1)
        key, order = torch.sort(key)
        prod = (av[ea] * bv[eb])[order]
        del ea, eb, order
        key, inv = torch.unique_consecutive(key, return_inverse=True)
        vals.append(torch.zeros(key.numel(), dtype=torch.float64, device=DEV).index_add_(0, inv, prod))
        lens.append(torch.bincount(key // B.ncols - r0, minlength=r1 - r0))
        cols.append((key % B.ncols).to(torch.int32))
        del inv, prod, key
    rp = torch.zeros(A.nrows + 1, dtype=torch.int64, device=DEV)
    torch.cumsum(torch.cat(lens), 0, out=rp[1:])
    return sg.Csr(A.nrows, B.ncols, rp, torch.cat(cols), torch.cat(vals))


def _exact_gradients(A, B, C, dC):
    av, bv, g = A.val.detach().double(), B.val.detach().double(), dC.double()
    ckey = _row_ids(C) * C.ncols + C.col.to(torch.int64)
    dA, dB = torch.zeros_like(av), torch.zeros_like(bv)
    for r0, r1 in _row_blocks(A, B):
        ea, eb, key = _expand(A, B, r0, r1)
        t = g[torch.searchsorted(ckey, key)]
        dA.index_add_(0, ea, t * bv[eb])
        dB.index_add_(0, eb, t * av[ea])
    return [dA, dB]


def exact(case, seed):
    kind = case["kind"]
    if kind == "triangles":
        return None   # a whole number
    out, C = [], None
    if kind == "batched":
        parts = [_exact_product(a, b) for a, b in _operands(case, seed)]
        return [None, None, torch.cat([m.val for m in parts])]
    for A, B in _operands(case, seed):
        C = _exact_product(A, C if B is None else B)
        out += [None, None, C.val]
        if kind == "autograd":
            out += _exact_gradients(A, B, C, _upstream(C.nnz, A.val.dtype, seed))
    return out
