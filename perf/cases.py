"""Timing cases of the sparse-product library: inputs, one pass through the
public entry points (paper_2303_02471_gb300.ops / .autograd), the work a pass
cannot do without, and its result in 64 bits.

The matrices are the repository's own workloads (the 5-point Laplacian, the
uniformly random very sparse product, the R-MAT power law, the uneven batch,
the Galerkin product) drawn on the GPU, over the sizes that the tests and the
benchmark use and between them.  A case fixes the base patterns, so that every
seed gives outputs of the same sizes; the seed turns the indices of the
irregular ones (a rotation, the same for both sides of a contraction) and
draws the values.
"""
import math

import numpy as np
import torch

from paper_2303_02471_gb300 import autograd, ops

DEV = "cuda"
DTYPES = {"f64": torch.float64, "f32": torch.float32}


# ------------------------------------------------------------------- cases
def listed():
    return [
        # The smallest call: a stencil matrix squared (multigrid on a coarse
        # level, a unit of a larger solver). Launches and latency count.
        {"name": "stencil_32", "kind": "product", "matrix": "lap2d", "n": 32, "dtype": "f64"},
        # The very sparse product, 2^20 columns of 1 to 8 entries: the light
        # columns at full size, both phases.
        {"name": "random_1m", "kind": "product", "matrix": "random", "m": 1 << 20, "k": 1 << 20, "n": 1 << 20,
         "zmin": 1, "zmax": 8, "dtype": "f64"},
        # The power-law product (a graph squared), columns of every weight up
        # to hundreds of thousands of products: the headline, both phases.
        {"name": "rmat_18", "kind": "product", "matrix": "rmat", "n": 18, "dtype": "f64"},
        # A power-law graph in single precision.
        {"name": "rmat_16_f32", "kind": "product", "matrix": "rmat", "n": 16, "dtype": "f32"},
        # A rectangular product of odd sizes and mid-weight columns (a chain
        # A_1 A_2 of transfer or feature matrices), both phases.
        {"name": "ragged_12k", "kind": "product", "matrix": "random", "m": 12007, "k": 9973, "n": 15013,
         "zmin": 7, "zmax": 40, "dtype": "f64"},
        # New values on a known pattern (time stepping, Newton steps): the
        # numeric phase alone with a kept plan.
        {"name": "renumeric_rmat_17", "kind": "numeric", "matrix": "rmat", "n": 17, "dtype": "f64"},
        # The gradients of a product on its patterns (one layer's backward).
        {"name": "backward_rmat_16", "kind": "backward", "matrix": "rmat", "n": 16, "dtype": "f64"},
        # The form without a symbolic phase, on light columns, in single
        # precision, with a size that is no power of two.
        {"name": "single_pass_300k_f32", "kind": "single_pass", "matrix": "random", "m": 300007, "k": 300007,
         "n": 300007, "zmin": 1, "zmax": 8, "dtype": "f32"},
        # Row-major users: the CSR form of a mid-sized product.
        {"name": "csr_60k", "kind": "csr", "matrix": "random", "m": 60001, "k": 60001, "n": 60001, "zmin": 2,
         "zmax": 24, "dtype": "f64"},
        # A training step through the Galerkin product P^T (A P) at 40^3:
        # transpose, two products, their backward through autograd.
        {"name": "galerkin_40", "kind": "galerkin", "n": 40, "dtype": "f64"},
        # Uneven products of both precisions as one batch, both phases, with
        # the thresholds that the batch autotuner picks for them.
        {"name": "batch_28", "kind": "batch", "count": 28, "lo": 500, "hi": 20000, "zmin": 2, "zmax": 40,
         "tuned": True},
        # A training step of a batch (forward and backward) with the default
        # configuration and smaller products.
        {"name": "batch_train_12", "kind": "batch_train", "count": 12, "lo": 300, "hi": 4000, "zmin": 2, "zmax": 24,
         "tuned": False},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["product", "product", "product", "numeric", "backward", "single_pass", "csr", "galerkin",
                       "batch", "batch_train"])
    if kind == "galerkin":
        return {"kind": kind, "n": 2 * rng.randint(8, 24), "dtype": "f64"}
    if kind in ("batch", "batch_train"):
        lo = rng.randint(100, 800)
        hi = _log_int(rng, 1000, 20000 if kind == "batch" else 6000)
        return {"kind": kind, "count": rng.randint(3, 28 if kind == "batch" else 12), "lo": lo, "hi": hi, "zmin": 2,
                "zmax": rng.randint(4, 40 if kind == "batch" else 24), "tuned": rng.random() < 0.5}
    dtype = rng.choice(["f64", "f64", "f32"])
    what = rng.choice(["random", "random", "rmat"] + (["lap2d"] if kind in ("product", "numeric") else []))
    if what == "lap2d":
        return {"kind": kind, "matrix": what, "n": _log_int(rng, 8, 700), "dtype": dtype}
    if what == "rmat":
        # the edge factor varies too, so that drawn graphs differ
        return {"kind": kind, "matrix": what, "n": rng.randint(9, 17), "edges": rng.randint(4, 10), "dtype": dtype}
    n = _log_int(rng, 500, 1 << 20)
    # products: about n * z^2, at most some 30 million
    top = min(40.0, math.sqrt(3.0e7 / n) * 1.6)
    zmax = max(2, int(round(math.exp(rng.uniform(math.log(2.0), math.log(max(2.1, top)))))))
    m, k = (max(zmax, int(n * rng.uniform(0.6, 1.6))) for _ in range(2))
    return {"kind": kind, "matrix": what, "m": m, "k": k, "n": n, "zmin": rng.randint(1, max(1, zmax // 2)),
            "zmax": zmax, "dtype": dtype}


# ------------------------------------------------------------------ inputs
def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _turned(nrows, ncols, key, rshift, cshift):
    """The keys with rows and columns rotated, ascending."""
    return ((key // nrows + cshift) % ncols * nrows + (key % nrows + rshift) % nrows).sort().values


def _from_keys(nrows, ncols, key, values):
    """CSC arrays of ascending distinct keys col * nrows + row."""
    counts = torch.bincount(key // nrows, minlength=ncols)
    colptr = torch.zeros(ncols + 1, dtype=torch.int64, device=DEV)
    torch.cumsum(counts, 0, out=colptr[1:])
    return ops.CscMatrix(nrows, ncols, colptr, (key % nrows).to(torch.int32), values)


def _random(nrows, ncols, zmin, zmax, g):
    """Keys of Z ~ U{zmin..zmax} distinct uniform rows per column."""
    zmax = min(zmax, nrows)
    z = torch.randint(min(zmin, zmax), zmax + 1, (ncols, 1), generator=g, device=DEV)
    rows = torch.randint(0, nrows, (ncols, zmax), generator=g, device=DEV)
    rows[torch.arange(zmax, device=DEV)[None, :] >= z] = nrows  # no entry
    while True:
        rows = rows.sort(dim=1).values
        again = torch.zeros_like(rows, dtype=torch.bool)
        again[:, 1:] = (rows[:, 1:] == rows[:, :-1]) & (rows[:, 1:] < nrows)
        count = int(again.sum())
        if count == 0:
            break
        rows[again] = torch.randint(0, nrows, (count,), generator=g, device=DEV)
    return (rows + nrows * torch.arange(ncols, device=DEV)[:, None])[rows < nrows]


def _random_pair(m, k, n, zmin, zmax, dtype, base, seed):
    """A (m x k) and B (k x n) with N(0, 1) values."""
    g, s = _gen(base), _gen(seed)
    ra, rk, rb = (int(torch.randint(0, size, (1,), generator=s, device=DEV)) for size in (m, k, n))
    ka = _turned(m, k, _random(m, k, zmin, zmax, g), ra, rk)
    kb = _turned(k, n, _random(k, n, zmin, zmax, g), rk, rb)
    return tuple(_from_keys(rows, cols, key, torch.randn(key.numel(), generator=s, device=DEV, dtype=dtype))
                 for rows, cols, key in ((m, k, ka), (k, n, kb)))


def _rmat(scale, edges, dtype, seed, cap=2000):
    """R-MAT (0.57, 0.19, 0.19, 0.05), `edges` per column drawn, duplicates
    dropped, at most `cap` entries per column, U[-1, 1] values."""
    n = 1 << scale
    g = _gen(scale)
    row = torch.zeros(edges * n, dtype=torch.int64, device=DEV)
    col = torch.zeros_like(row)
    for _ in range(scale):
        u = torch.rand(edges * n, generator=g, device=DEV, dtype=torch.float64)
        row = 2 * row + (u >= 0.76)
        col = 2 * col + (((u >= 0.57) & (u < 0.76)) | (u >= 0.95))
    key = torch.unique(col * n + row)
    # a random subset of `cap` entries of every longer column
    mix = torch.rand(key.numel(), generator=g, device=DEV, dtype=torch.float64)
    c = key // n
    order = torch.argsort(c.to(torch.float64) + mix)
    start = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
    torch.cumsum(torch.bincount(c, minlength=n), 0, out=start[1:])
    rank = torch.arange(key.numel(), device=DEV) - start[c[order]]
    s = _gen(seed)
    shift = int(torch.randint(0, n, (1,), generator=s, device=DEV))
    key = _turned(n, n, key[order[rank < cap]], shift, shift)
    return _from_keys(n, n, key, torch.rand(key.numel(), generator=s, device=DEV, dtype=dtype) * 2 - 1)


def _stencil(g, dims):
    """Keys of the (2 dims + 1)-point Laplacian of a g^dims grid and which of
    them lie on the diagonal."""
    n = g ** dims
    idx = torch.arange(n, device=DEV)
    keys, diag = [idx * n + idx], [torch.ones(n, dtype=torch.bool, device=DEV)]
    for d in range(dims):
        x = (idx // g ** d) % g
        for s in (-1, 1):
            on = idx[(x + s >= 0) & (x + s < g)]
            keys.append(on * n + on + s * g ** d)
            diag.append(torch.zeros(on.numel(), dtype=torch.bool, device=DEV))
    key, order = torch.cat(keys).sort()
    return n, key, torch.cat(diag)[order]


def _lap2d(g_side, dtype, g):
    n, key, _ = _stencil(g_side, 2)
    return _from_keys(n, n, key, torch.rand(key.numel(), generator=g, device=DEV, dtype=dtype) * 2 - 1)


def _lap3d(g_side):
    n, key, diag = _stencil(g_side, 3)
    return _from_keys(n, n, key, torch.where(diag, 6.0, -1.0).to(torch.float64))


def _prolongation(g_side, seed):
    """g^3 x (g/2)^3 aggregation: every row in its aggregate, half of the rows
    in a neighbouring one too, values U[0.5, 1]."""
    g = _gen(g_side)
    h, n = g_side // 2, g_side ** 3
    idx = torch.arange(n, device=DEV)
    ac = torch.stack([(idx // g_side ** d) % g_side // 2 for d in range(3)])
    agg = ac[0] + h * ac[1] + h * h * ac[2]
    axis = torch.randint(0, 3, (n,), generator=g, device=DEV)
    sign = torch.randint(0, 2, (n,), generator=g, device=DEV) * 2 - 1
    at = ac.gather(0, axis[None])[0]
    sign = torch.where((at + sign < 0) | (at + sign >= h), -sign, sign)
    agg2 = agg + sign * torch.tensor([1, h, h * h], device=DEV)[axis]
    two = torch.rand(n, generator=g, device=DEV) < 0.5
    key = torch.cat([agg * n + idx, agg2[two] * n + idx[two]]).sort().values
    return _from_keys(n, h ** 3, key,
                      0.5 + 0.5 * torch.rand(key.numel(), generator=_gen(seed), device=DEV, dtype=torch.float64))


def _pair(case, seed):
    """The operands of one product (A and B are the same matrix when square
    graphs and stencils are squared)."""
    dtype = DTYPES[case["dtype"]]
    if case["matrix"] == "lap2d":
        A = _lap2d(case["n"], dtype, _gen(seed))
        return A, A
    if case["matrix"] == "rmat":
        A = _rmat(case["n"], case.get("edges", 8), dtype, seed)
        return A, A
    return _random_pair(case["m"], case["k"], case["n"], case["zmin"], case["zmax"], dtype, case["n"], seed)


def _batch(case, seed):
    """Uneven square pairs: sizes log-uniform, entries per column uniform in
    zmin..zmax and constant in a matrix, the first half in double precision,
    the second in single."""
    sizes = np.random.default_rng(case["count"])
    As, Bs = [], []
    for i in range(case["count"]):
        n = int(round(math.exp(sizes.uniform(math.log(case["lo"]), math.log(case["hi"])))))
        z = int(sizes.integers(case["zmin"], case["zmax"] + 1))
        dtype = torch.float64 if i < case["count"] // 2 else torch.float32
        A, B = _random_pair(n, n, n, z, z, dtype, i, seed + i)
        As.append(A)
        Bs.append(B)
    return As, Bs


def _galerkin_inputs(case, seed):
    """A, P and the target's values on the pattern of P^T (A P): a product of
    nearby values, perturbed by up to one per cent."""
    A, P = _lap3d(case["n"]), _prolongation(case["n"], seed)
    C = _galerkin64(A, P)[0]
    noise = torch.rand(C["values"].numel(), generator=_gen(seed + 1), device=DEV, dtype=torch.float64) * 2 - 1
    return A, P, C["values"] * (1 + 0.01 * noise)


def _config(case):
    # t and the CTA size are what the batch autotuner finds for such batches
    return ops.Config(t=33, cta_threads=128) if case["tuned"] else ops.Config()


# -------------------------------------------------------------------- passes
def prepare(case, seed):
    kind = case["kind"]
    if kind == "galerkin":
        A, P, T = _galerkin_inputs(case, seed)
        return {"kind": kind, "A": A, "P": P, "T": T}
    if kind in ("batch", "batch_train"):
        As, Bs = _batch(case, seed)
        state = {"kind": kind, "As": As, "Bs": Bs, "config": _config(case)}
        if kind == "batch_train":
            g = _gen(seed + 1)
            plan = ops.spgemm_batched_symbolic(As, Bs, state["config"])
            state["dCs"] = [torch.randn(n, generator=g, device=DEV, dtype=A.dtype) for n, A in zip(plan.nnz, As)]
            plan.destroy()
        return state
    A, B = _pair(case, seed)
    if kind == "csr":
        # the CSR arrays of A B are the CSC arrays of (B^T A^T): the operands
        # swap places
        rows = [ops.CsrMatrix(M.ncols, M.nrows, M.colptr, M.rowidx, M.values) for M in (B, A)]
        return {"kind": kind, "A": rows[0], "B": rows[1]}
    state = {"kind": kind, "A": A, "B": B}
    if kind == "numeric":
        state["plan"] = ops.spgemm_symbolic(A, B)[2]
    elif kind == "backward":
        state["C"], state["plan"] = ops.spgemm(A, B)
        state["dC"] = torch.randn(state["C"].nnz, generator=_gen(seed + 1), device=DEV, dtype=A.dtype)
    return state


def run(s):
    kind = s["kind"]
    if kind == "product":
        C, _ = ops.spgemm(s["A"], s["B"])
        return C.colptr, C.rowidx, C.values
    if kind == "numeric":
        C = ops.spgemm_numeric(s["plan"], s["A"], s["B"])
        return C.colptr, C.rowidx, C.values
    if kind == "backward":
        return ops.spgemm_backward(s["plan"], s["A"], s["B"], s["C"], s["dC"])
    if kind == "single_pass":
        C, _ = ops.spgemm_single_pass(s["A"], s["B"])
        return C.colptr, C.rowidx, C.values
    if kind == "csr":
        C, _ = ops.spgemm_csr(s["A"], s["B"])
        return C.rowptr, C.colidx, C.values
    if kind == "galerkin":
        p = s["P"].values.detach().requires_grad_()
        C = autograd.galerkin(s["A"], s["P"].with_values(p))
        loss = (C.values - s["T"]).square().sum()
        loss.backward()
        return C.colptr, C.rowidx, C.values.detach(), p.grad
    Cs, plan = ops.spgemm_batched(s["As"], s["Bs"], s["config"])
    out = [plan.colptr, [C.rowidx for C in Cs], [C.values for C in Cs]]
    if kind == "batch_train":
        out += ops.spgemm_batched_backward(plan, s["As"], s["Bs"], Cs, s["dCs"])
    return out


# ---------------------------------------------------------------- references
def _expand(A, B, p0, p1):
    """The products of B's entries [p0, p1): the positions in A and in B."""
    k = B.rowidx[p0:p1].long()
    z = A.colptr[k + 1] - A.colptr[k]
    pb = torch.repeat_interleave(torch.arange(p0, p1, device=DEV), z)
    first = torch.repeat_interleave(A.colptr[k] - (torch.cumsum(z, 0) - z), z)
    return first + torch.arange(pb.numel(), device=DEV), pb


def _columns(M):
    return torch.repeat_interleave(torch.arange(M.ncols, device=DEV), torch.diff(M.colptr))


def _chunks(A, B, most=1 << 26):
    """Column ranges of B of about `most` products each."""
    k = B.rowidx.long()
    ops_before = torch.zeros(B.nnz + 1, dtype=torch.int64, device=DEV)
    torch.cumsum(A.colptr[k + 1] - A.colptr[k], 0, out=ops_before[1:])
    at = ops_before[B.colptr].cpu().numpy()
    j = 0
    while j < B.ncols:
        e = max(j + 1, int(np.searchsorted(at, at[j] + most, side="right")) - 1)
        yield j, min(e, B.ncols), int(at[min(e, B.ncols)] - at[j])
        j = e


def _product64(A, B, av=None, bv=None):
    """C = A B in 64 bits: colptr, rowidx and values."""
    av = A.values.double() if av is None else av
    bv = B.values.double() if bv is None else bv
    cols, rows, values = _columns(B), [], []
    counts = torch.zeros(B.ncols, dtype=torch.int64, device=DEV)
    for j0, j1, _ in _chunks(A, B):
        p0, p1 = int(B.colptr[j0]), int(B.colptr[j1])
        qa, pb = _expand(A, B, p0, p1)
        key, order = (cols[pb] * A.nrows + A.rowidx[qa]).sort(stable=True)
        terms = (av[qa] * bv[pb])[order]
        key, place = torch.unique_consecutive(key, return_inverse=True)
        values.append(torch.zeros(key.numel(), dtype=torch.float64, device=DEV).index_add_(0, place, terms))
        rows.append((key % A.nrows).to(torch.int32))
        counts += torch.bincount(key // A.nrows, minlength=B.ncols)
    colptr = torch.zeros(B.ncols + 1, dtype=torch.int64, device=DEV)
    torch.cumsum(counts, 0, out=colptr[1:])
    none = torch.zeros(0, device=DEV)
    return {"colptr": colptr, "rowidx": torch.cat(rows) if rows else none.int(),
            "values": torch.cat(values) if values else none.double()}


def _gradients64(A, B, C, dC, av=None, bv=None):
    """dA and dB on the stored entries, in 64 bits; C as _product64 gives it."""
    av = A.values.double() if av is None else av
    bv = B.values.double() if bv is None else bv
    dC = dC.double()
    ccol = torch.repeat_interleave(torch.arange(B.ncols, device=DEV), torch.diff(C["colptr"]))
    ckey, cols = ccol * A.nrows + C["rowidx"], _columns(B)
    dA, dB = (torch.zeros(M.nnz, dtype=torch.float64, device=DEV) for M in (A, B))
    for j0, j1, _ in _chunks(A, B):
        p0, p1 = int(B.colptr[j0]), int(B.colptr[j1])
        qa, pb = _expand(A, B, p0, p1)
        d = dC[torch.searchsorted(ckey, cols[pb] * A.nrows + A.rowidx[qa])]
        dA.index_add_(0, qa, bv[pb] * d)
        dB.index_add_(0, pb, av[qa] * d)
    return dA, dB


def _transposed(M):
    """M^T and the permutation of its values."""
    key, perm = (M.rowidx.long() * M.ncols + _columns(M)).sort()
    return _from_keys(M.ncols, M.nrows, key, M.values[perm]), perm


def _galerkin64(A, P):
    """P^T (A P) with what its gradient needs."""
    M = _product64(A, P)
    Mm = ops.CscMatrix(A.nrows, P.ncols, M["colptr"], M["rowidx"], M["values"])
    Pt, perm = _transposed(P)
    return _product64(Pt, Mm), M, Mm, Pt, perm


def exact(case, seed):
    kind = case["kind"]
    if kind == "galerkin":
        A, P, T = _galerkin_inputs(case, seed)
        C, M, Mm, Pt, perm = _galerkin64(A, P)
        dPt, dM = _gradients64(Pt, Mm, C, 2 * (C["values"] - T))
        dP = _gradients64(A, P, M, dM)[1]
        dP[perm] += dPt
        return C["colptr"], C["rowidx"], C["values"], dP
    if kind in ("batch", "batch_train"):
        As, Bs = _batch(case, seed)
        Cs = [_product64(A, B) for A, B in zip(As, Bs)]
        out = [torch.cat([C["colptr"] for C in Cs]), [C["rowidx"] for C in Cs], [C["values"] for C in Cs]]
        if kind == "batch_train":
            g = _gen(seed + 1)
            dCs = [torch.randn(C["values"].numel(), generator=g, device=DEV, dtype=A.dtype)
                   for C, A in zip(Cs, As)]
            grads = [_gradients64(A, B, C, d) for A, B, C, d in zip(As, Bs, Cs, dCs)]
            out += [[dA for dA, _ in grads], [dB for _, dB in grads]]
        return out
    A, B = _pair(case, seed)
    C = _product64(A, B)
    if kind == "backward":
        dC = torch.randn(C["values"].numel(), generator=_gen(seed + 1), device=DEV, dtype=A.dtype)
        return _gradients64(A, B, C, dC)
    return C["colptr"], C["rowidx"], C["values"]


# ---------------------------------------------------------------------- work
def _bytes(M):
    return M.colptr.numel() * 8 + M.nnz * (4 + M.dtype.itemsize)


def _product_work(A, B, backward=False, forward=True):
    """Inputs once, outputs once; two operations per product, twice as many
    backward (a product for dA and one for dB)."""
    products = nnz = 0
    cols = _columns(B)
    for j0, j1, count in _chunks(A, B):
        qa, pb = _expand(A, B, int(B.colptr[j0]), int(B.colptr[j1]))
        nnz += torch.unique(cols[pb] * A.nrows + A.rowidx[qa]).numel()
        products += count
    w = A.dtype.itemsize
    inputs = _bytes(A) + (0 if B is A else _bytes(B))
    pattern = 8 * (B.ncols + 1) + nnz * 4
    total, flops = inputs, 0
    if forward:
        total += pattern + nnz * w
        flops += 2 * products
    if backward:  # dC in, dA and dB out; the pattern too when it is not made here
        total += nnz * w + (A.nnz + B.nnz) * w + (0 if forward else pattern)
        flops += 4 * products
    return total, flops


def work(case):
    kind = case["kind"]
    if kind == "galerkin":
        A, P, T = _galerkin_inputs(case, 0)
        _, _, Mm, Pt, _ = _galerkin64(A, P)
        products = sum(c for X, Y in ((A, P), (Pt, Mm)) for _, _, c in _chunks(X, Y))
        return {"bytes": _bytes(A) + _bytes(P) + T.numel() * (8 + 4 + 8) + 8 * (P.ncols + 1) + P.nnz * 8,
                "flops": 6 * products}
    if kind in ("batch", "batch_train"):
        parts = [_product_work(A, B, backward=kind == "batch_train") for A, B in zip(*_batch(case, 0))]
    else:
        A, B = _pair(case, 0)
        parts = [_product_work(A, B, backward=kind == "backward", forward=kind != "backward")]
    return {"bytes": sum(b for b, _ in parts), "flops": sum(f for _, f in parts)}
