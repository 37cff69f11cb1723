"""The preparation of a product on the GPU: Op_j, bins, row compaction and the
checks of both operands, at the edges of its tiles and runs."""
import numpy as np
import pytest

import oracle
from paper_2303_02471_gb300 import synth

from gpu_helpers import assert_matches_oracle, upload

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def _matrix(rng, nrows, lengths, rows=None):
    """Columns of the given lengths with distinct rows out of `rows`."""
    rows = np.arange(nrows) if rows is None else rows
    cp = np.concatenate([[0], np.cumsum(lengths)]).astype(np.int64)
    idx = [rng.permutation(rows)[:z] for z in lengths]
    idx = np.concatenate(idx + [np.zeros(0)]).astype(np.int32)
    return synth.CSC(nrows, len(lengths), cp, idx, rng.standard_normal(idx.size))


@pytest.mark.parametrize("n", [1, 3, 4, 5, 31, 129, 2501])
@pytest.mark.parametrize("m", [7, 2047, 2049, 8 * 2048 + 1, 9 * 2048])
def test_counts_and_compact_rows(m, n):
    """Columns of B at the edge between a lane's and a warp's count; rows of A
    with entries in some rows only (renumbered) or in all but one."""
    from paper_2303_02471_gb300 import ops
    rng = np.random.default_rng(m + n)
    k = 600
    for rows in (np.arange(0, m, 3), np.arange(m - 1)):
        A = _matrix(rng, m, rng.integers(0, min(6, rows.size) + 1, k), rows)
        B = _matrix(rng, k, np.array([[0, 1, 24, 25, 3, 255, 2, 257, 600][i % 9] for i in range(n)]))
        C, plan = ops.spgemm(upload(A), upload(B))
        za = np.diff(A.colptr)
        op = np.add.reduceat(np.append(za[B.rowidx], 0), B.colptr[:-1]) * (np.diff(B.colptr) > 0)
        assert np.array_equal(plan.op_counts().cpu().numpy(), op)
        assert plan.info()["products"] == op.sum()
        assert_matches_oracle(C, A, B)
        plan.check()


@pytest.mark.parametrize("what", ["row_short", "row_long", "row_negative", "colptr_falls", "colptr_beyond", "colptr_end",
                                  "colptr_start", "no_columns", "a_row", "a_colptr"])
def test_malformed_operands_are_rejected(what):
    """Every malformed operand is an error of the call (nothing follows it),
    and the next product is right."""
    import torch
    from paper_2303_02471_gb300 import ops
    rng = np.random.default_rng(5)
    A = _matrix(rng, 400, rng.integers(1, 8, 300))
    B = _matrix(rng, 300, np.array([3, 40, 0, 200, 5, 1, 24, 25]))
    dA, dB = upload(A), upload(B)
    bad = ops.CscMatrix(dB.nrows, dB.ncols, dB.colptr.clone(), dB.rowidx.clone(), dB.values)
    badA = ops.CscMatrix(dA.nrows, dA.ncols, dA.colptr.clone(), dA.rowidx.clone(), dA.values)
    if what == "row_short":
        bad.rowidx[1] = 300
    elif what == "row_long":
        bad.rowidx[100] = 2000000000
    elif what == "row_negative":
        bad.rowidx[-1] = -1
    elif what == "colptr_falls":
        bad.colptr[3] = 1
    elif what == "colptr_beyond":
        bad.colptr[4] = 1 << 40
    elif what == "colptr_end":
        bad.colptr[-1] -= 1
    elif what == "colptr_start":
        bad.colptr[0] = 1
    elif what == "no_columns":
        bad = ops.CscMatrix(300, 0, torch.zeros(1, dtype=torch.int64, device="cuda"), dB.rowidx, dB.values)
    elif what == "a_row":
        badA.rowidx[7] = 400
    else:
        badA.colptr[5] = badA.colptr[4] - 1
    with pytest.raises(RuntimeError, match="SPG_ERR_INVALID"):
        if what.startswith("a_"):
            ops.spgemm(badA, dB)
        else:
            ops.spgemm(dA, bad)
    C, plan = ops.spgemm(dA, dB)
    plan.check()
    assert_matches_oracle(C, A, B)


@pytest.mark.parametrize("heavy", [1, 5, 700])
def test_dense_list_from_both_ends(heavy):
    """Columns of every weight class in the dense bin, `heavy` of them far
    heavier than the rest, forward and backward: each column is worked once."""
    import torch
    from paper_2303_02471_gb300 import ops
    rng = np.random.default_rng(heavy)
    A = _matrix(rng, 2000, rng.integers(0, 60, 900))
    n = 1500
    B = _matrix(rng, 900, np.where(np.arange(n) % max(1, n // heavy) == 3, 800, rng.integers(0, 12, n)))
    dA, dB = upload(A), upload(B)
    C, plan = ops.spgemm(dA, dB, ops.Config(t=1))
    assert_matches_oracle(C, A, B)
    dc = torch.as_tensor(rng.standard_normal(C.nnz), device="cuda")
    got = ops.spgemm_backward(plan, dA, dB, C, dc)
    plan.check()
    Ch, d = C.to_host(), dc.cpu().numpy()
    want = oracle.backward(A, B, Ch, d)
    scale = oracle.backward(A.with_values(np.abs(A.values)), B.with_values(np.abs(B.values)), Ch, np.abs(d))
    for g, r, s in zip(got, want, scale):  # sums of at most 2000 terms: 2.2e-13 of their size
        assert np.all(np.abs(g.cpu().numpy() - r) <= 1e-12 * s)


@pytest.mark.parametrize("what", ["row", "colptr", "a_rows_unchecked"])
def test_malformed_operands_of_many_ctas(what):
    """A fault that some CTAs report while others start (several waves of
    them): every CTA takes the whole decision, and the next product is right."""
    import torch
    from paper_2303_02471_gb300 import ops
    rng = np.random.default_rng(11)
    n = 400003
    A = _matrix(rng, 900, rng.integers(1, 5, 300), np.arange(0, 900, 3))
    B = _matrix(rng, 300, np.where(np.arange(1000) % 50 == 0, 60, rng.integers(0, 4, 1000)))
    # the 1000 columns over and over
    reps = -(-n // 1000)
    cp = (np.arange(reps)[:, None] * B.nnz + B.colptr[None, :-1]).ravel()
    cp = np.append(cp, reps * B.nnz)
    big = synth.CSC(300, reps * 1000, cp, np.tile(B.rowidx, reps), np.tile(B.values, reps))
    dA, dB = upload(A), upload(big)
    bad = ops.CscMatrix(dB.nrows, dB.ncols, dB.colptr.clone(), dB.rowidx.clone(), dB.values)
    badA = ops.CscMatrix(dA.nrows, dA.ncols, dA.colptr, dA.rowidx.clone(), dA.values)
    if what == "row":
        bad.rowidx[3::50021] = 300
    elif what == "colptr":
        bad.colptr[1::10007] = -1
    else:  # rows out of range without validation: found by the renumbering
        badA.rowidx[::7] = 900
    for _ in range(3):
        with pytest.raises(RuntimeError, match="SPG_ERR_INVALID"):
            if what.startswith("a_"):
                ops.spgemm_symbolic(badA, dB, ops.Config(validate=False))
            else:
                ops.spgemm_symbolic(dA, bad)
    C, plan = ops.spgemm(dA, upload(B))
    plan.check()
    assert_matches_oracle(C, A, B)


def test_rows_of_many_tiles():
    """Row tiles at and past the number up to which every CTA adds up the
    tiles' counts itself: the same rows, numbered with one launch more."""
    from paper_2303_02471_gb300 import ops
    rng = np.random.default_rng(3)
    k, n = 3000, 200
    za = rng.integers(1, 7, k)
    launches = []
    B = _matrix(rng, k, rng.integers(0, 40, n))
    for tiles in (4096, 4097, 4096 + 8193):  # the last: more than one step of the prefix sums
        m = tiles * 2048 - 5
        cp = np.concatenate([[0], np.cumsum(za)]).astype(np.int64)
        rows = np.concatenate([np.arange(z) * (m // z) + rng.integers(0, m // z, z) for z in za])
        rows[0], rows[-1] = 0, m - 1  # the first and the last tile
        A = synth.CSC(m, k, cp, rows.astype(np.int32), rng.standard_normal(rows.size))
        C, plan = ops.spgemm(upload(A), upload(B))
        plan.check()
        assert_matches_oracle(C, A, B)
        launches.append(plan.launch_count()["symbolic"])
    assert launches[1] == launches[2] == launches[0] + 1
