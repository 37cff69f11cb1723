"""The single pass's two-call form (begin, finish) and what its plans and its
operands must satisfy."""
import ctypes

import numpy as np
import pytest

from paper_2303_02471_gb300 import synth

from gpu_helpers import assert_matches_oracle, upload

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def _ptr(t):
    return ctypes.c_void_p(t.data_ptr())


@pytest.mark.parametrize("handle", [True, False])
def test_unfinished_plan_serves_no_product(handle):
    """Before finish, and after a finish that failed, numeric, backward and
    copy are refused; once finished the plan serves all three."""
    import torch
    from paper_2303_02471_gb300 import _native as N
    from paper_2303_02471_gb300 import ops
    host = synth.rmat(9, seed=3, col_cap=100)
    A = upload(host)
    lib, s = N.lib(), ops._stream()
    cA = ops._csc(A)
    ref = ctypes.byref(cA)
    cfg = ops.Config(dense_cache_bytes=0).native()
    ws = torch.empty(ops.workspace_size(A, A, ops.Config(dense_cache_bytes=0)), dtype=torch.uint8, device="cuda")
    cp = torch.empty(A.ncols + 1, dtype=torch.int64, device="cuda")
    want, _ = ops.spgemm(A, A)
    rows = torch.empty(want.nnz, dtype=torch.int32, device="cuda")
    vals = torch.empty(want.nnz, dtype=torch.float64, device="cuda")
    grad = torch.empty(A.nnz, dtype=torch.float64, device="cuda")
    need, h, nnz = ctypes.c_size_t(), ctypes.c_void_p(), ctypes.c_int64()
    assert lib.spgemm_single_pass_begin(ops.handle().ptr if handle else None, ref, ref, ctypes.byref(cfg), _ptr(ws),
                                        ws.numel(), _ptr(cp), ctypes.byref(need), ctypes.byref(h), s) == 0

    def uses():
        return [lib.spgemm_numeric(h, ref, ref, _ptr(want.colptr), _ptr(rows), _ptr(vals), s),
                lib.spgemm_numeric(h, ref, ref, _ptr(want.colptr), None, None, s),
                lib.spgemm_backward(h, ref, ref, _ptr(want.colptr), _ptr(want.rowidx), _ptr(vals), _ptr(grad),
                                    _ptr(grad), s),
                lib.spgemm_single_pass_copy(h, _ptr(want.colptr), _ptr(rows), _ptr(vals), s)]

    assert [N.STATUS[x] for x in uses()] == ["SPG_ERR_INVALID"] * 4
    slots = torch.empty(need.value, dtype=torch.uint8, device="cuda")
    assert N.STATUS[lib.spgemm_single_pass_finish(h, ref, ref, _ptr(slots), need.value - 1, _ptr(cp),
                                                  ctypes.byref(nnz), s)] == "SPG_ERR_WORKSPACE"
    assert [N.STATUS[x] for x in uses()] == ["SPG_ERR_INVALID"] * 4
    assert lib.spgemm_single_pass_finish(h, ref, ref, _ptr(slots), need.value, _ptr(cp), ctypes.byref(nnz), s) == 0
    assert nnz.value == want.nnz and torch.equal(cp, want.colptr)
    # once per plan
    assert N.STATUS[lib.spgemm_single_pass_finish(h, ref, ref, _ptr(slots), need.value, _ptr(cp), ctypes.byref(nnz),
                                                  s)] == "SPG_ERR_INVALID"
    for call in (lambda: lib.spgemm_single_pass_copy(h, _ptr(cp), _ptr(rows), _ptr(vals), s),
                 lambda: lib.spgemm_numeric(h, ref, ref, _ptr(cp), _ptr(rows), _ptr(vals), s)):
        rows.fill_(-1)
        vals.fill_(float("nan"))
        assert call() == 0
        assert_matches_oracle(ops.CscMatrix(A.nrows, A.ncols, cp, rows, vals), host, host)
    assert lib.spgemm_backward(h, ref, ref, _ptr(cp), _ptr(rows), _ptr(vals), _ptr(grad), None, s) == 0
    assert lib.spg_plan_check(h, s) == 0
    lib.spg_plan_destroy(h)


@pytest.mark.parametrize("form", ["single_pass", "single_pass_workspace", "csr"])
@pytest.mark.parametrize("a_is_double", [True, False])
def test_operands_of_two_dtypes_are_refused(form, a_is_double):
    """B's values are described by their own dtype, so that a B of the other
    one is an error of the call instead of being read as A's."""
    from paper_2303_02471_gb300 import ops
    host = synth.rmat(8, seed=4, col_cap=60)
    da, db = (np.float64, np.float32) if a_is_double else (np.float32, np.float64)
    A, B = upload(host, da), upload(host, db)
    if form == "csr":
        A, B = (ops.CsrMatrix(M.ncols, M.nrows, M.colptr, M.rowidx, M.values) for M in (A, B))
        call = ops.spgemm_csr
    elif form == "single_pass":
        call = ops.spgemm_single_pass
    else:
        import torch
        need = ops.single_pass_workspace_size(A, B)

        def call(a, b):
            return ops.spgemm_single_pass(a, b, workspace=torch.empty(need, dtype=torch.uint8, device="cuda"))
    with pytest.raises(RuntimeError, match="SPG_ERR_INVALID"):
        call(A, B)
    C, plan = call(A, A)
    plan.check()
    if form != "csr":
        assert_matches_oracle(C, host, host)


@pytest.mark.parametrize("acc", ["auto", "hash"])
@pytest.mark.parametrize("t", [None, 300, (1 << 63) - 1])
def test_backward_of_a_single_pass_plan_in_every_bin(t, acc):
    """The single pass counts no largest column per bin: the backward's hash
    tables are sized by what bounds the columns."""
    import oracle
    import torch
    from paper_2303_02471_gb300 import ops
    host = synth.rmat(11, seed=6, col_cap=300)
    A = upload(host)
    C, plan = ops.spgemm_single_pass(A, A, ops.Config(t=t, small_accumulator=acc))
    dc = torch.randn(C.nnz, dtype=torch.float64, device="cuda")
    got = ops.spgemm_backward(plan, A, A, C, dc)
    plan.check()
    Ch, d = C.to_host(), dc.cpu().numpy()
    want = oracle.backward(host, host, Ch, d)
    Ha = host.with_values(np.abs(host.values))
    scale = oracle.backward(Ha, Ha, Ch, np.abs(d))
    for g, r, s in zip(got, want, scale):
        assert np.all(np.abs(g.cpu().numpy() - r) <= 1e-12 * s)
