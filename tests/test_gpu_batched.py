"""Batched products (one persistent launch, CUDA-graph replay, autotuner)
against the per-matrix calls and the CPU oracle."""
import os

import numpy as np
import pytest

import oracle
from paper_2303_02471_gb300 import synth

from gpu_helpers import TAU, assert_matches_oracle, upload

pytestmark = pytest.mark.gpu

INF = (1 << 63) - 1
NCPU = len(os.sched_getaffinity(0))


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def _upload_pairs(pairs):
    return [upload(A) for A, _ in pairs], [upload(B) for _, B in pairs]


@pytest.mark.parametrize("t", [None, 0, 257, INF])
def test_batched_matches_oracle_and_plain(t):
    from paper_2303_02471_gb300 import ops
    pairs = synth.batch_pairs(24, seed=3, n_scale=0.05)
    As, Bs = _upload_pairs(pairs)
    cfg = ops.Config(t=t)
    Cs, plan = ops.spgemm_batched(As, Bs, cfg)
    plan.check()
    info = plan.info()
    assert info["launches"][1] == 1
    for (A, B), C, dA, dB in zip(pairs, Cs, As, Bs):
        assert_matches_oracle(C, A, B)
        P, pp = ops.spgemm(dA, dB, cfg)
        assert (P.colptr == C.colptr).all() and (P.rowidx == C.rowidx).all()


def test_batched_mixed_shapes_and_empty_products():
    from paper_2303_02471_gb300 import ops
    rng = np.random.default_rng(5)
    pairs = [synth.fuzz_pair(s) for s in range(12)]
    pairs += [(synth.random_pattern(rng, 300, 200, 0.05), synth.random_pattern(rng, 200, 150, 0.05))]
    As, Bs = _upload_pairs(pairs)
    Cs, plan = ops.spgemm_batched(As, Bs)
    plan.check()
    for (A, B), C in zip(pairs, Cs):
        assert_matches_oracle(C, A, B)


def test_batched_graph_replay():
    import torch
    from paper_2303_02471_gb300 import ops
    pairs = synth.batch_pairs(32, seed=4, n_scale=0.05)
    As, Bs = _upload_pairs(pairs)
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        plan = ops.spgemm_batched_symbolic(As, Bs)
        first = [(C.rowidx.clone(), C.values.clone()) for C in ops.spgemm_batched_numeric(plan, As, Bs, True)]
        for C in plan.outputs:
            C[0].zero_()
            C[1].zero_()
        Cs = ops.spgemm_batched_numeric(plan, As, Bs, True)  # replay
        plan.check()
    s.synchronize()
    refs = [oracle.spgemm(A, B) for A, B in pairs]
    for (A, B), C, (r0, v0), ref in zip(pairs, Cs, first, refs):
        assert (C.rowidx == r0).all()
        assert_matches_oracle(C, A, B, ref=ref)


def test_batched_graph_request_on_default_stream_launches_directly():
    # the legacy default stream cannot be captured; the launch still runs
    import torch
    from paper_2303_02471_gb300 import ops
    pairs = synth.batch_pairs(12, seed=8, n_scale=0.05)
    As, Bs = _upload_pairs(pairs)
    assert torch.cuda.current_stream().cuda_stream == 0
    plan = ops.spgemm_batched_symbolic(As, Bs)
    Cs = ops.spgemm_batched_numeric(plan, As, Bs, True)
    Cs = ops.spgemm_batched_numeric(plan, As, Bs, True)
    plan.check()
    for (A, B), C in zip(pairs, Cs):
        assert_matches_oracle(C, A, B)


@pytest.mark.parametrize("threads", [128, 256])
def test_batched_small_ctas_match_oracle(threads):
    from paper_2303_02471_gb300 import ops
    pairs = synth.batch_pairs(16, seed=9, n_scale=0.05)
    As, Bs = _upload_pairs(pairs)
    Cs, plan = ops.spgemm_batched(As, Bs, ops.Config(cta_threads=threads))
    plan.check()
    for (A, B), C in zip(pairs, Cs):
        assert_matches_oracle(C, A, B)


@pytest.mark.parametrize("tall", [False, True])
@pytest.mark.parametrize("t", [0, None])
def test_batched_dense_columns_per_warp_and_per_cta(tall, t):
    # flags of at most 1024 words: dense columns of the forward phases are
    # worked one per warp; a product with more than 32768 rows switches the
    # launch to one column per CTA
    from paper_2303_02471_gb300 import ops
    rng = np.random.default_rng(11)
    pairs = synth.batch_pairs(12, seed=10, n_scale=0.05)
    pairs += [(synth.random_pattern(rng, 2000, 90, 0.04, dtype=np.float32, dense_col=True),
               synth.random_pattern(rng, 90, 70, 0.3, dtype=np.float32))]
    if tall:
        pairs += [(synth.random_pattern(rng, 40000, 60, 0.002), synth.random_pattern(rng, 60, 40, 0.3))]
    As, Bs = _upload_pairs(pairs)
    Cs, plan = ops.spgemm_batched(As, Bs, ops.Config(t=t))
    plan.check()
    assert plan.info()["bins"][13] > 0
    for (A, B), C in zip(pairs, Cs):
        assert_matches_oracle(C, A, B)


@pytest.mark.parametrize("cache", [0, 4 * 700, None])
def test_batched_kept_dense_flags(cache):
    # dense columns one per warp keep their flags from the symbolic phase
    # for the numeric one: none kept, the first few columns, all of them
    import torch
    from paper_2303_02471_gb300 import ops
    pairs = synth.batch_pairs(20, seed=13, n_scale=0.05)
    As, Bs = _upload_pairs(pairs)
    cfg = ops.Config(t=0, dense_cache_bytes=cache)
    plan = ops.spgemm_batched_symbolic(As, Bs, cfg)
    assert plan.info()["bins"][13] > 0
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        first = [(C.rowidx.clone(), C.values.clone()) for C in ops.spgemm_batched_numeric(plan, As, Bs, True)]
        Cs = ops.spgemm_batched_numeric(plan, As, Bs, True)  # replay reads the kept flags again
    s.synchronize()
    plan.check()
    for (A, B), C, (r0, v0) in zip(pairs, Cs, first):
        assert (C.rowidx == r0).all()
        assert_matches_oracle(C, A, B)


def test_batched_backward_matches_plain():
    import torch
    from paper_2303_02471_gb300 import ops
    pairs = synth.batch_pairs(16, seed=6, n_scale=0.04)
    As, Bs = _upload_pairs(pairs)
    Cs, plan = ops.spgemm_batched(As, Bs)
    rng = np.random.default_rng(1)
    dCs = [torch.as_tensor(rng.standard_normal(C.nnz), device="cuda").to(C.values.dtype) for C in Cs]
    gA, gB = ops.spgemm_batched_backward(plan, As, Bs, Cs, dCs)
    plan.check()
    for (A, B), C, dc, ga, gb in zip(pairs, Cs, dCs, gA, gB):
        Ch = C.to_host()
        d = dc.cpu().numpy()
        rA, rB = oracle.backward(A, B, Ch, d)
        sA, sB = oracle.backward(A.with_values(np.abs(A.values)), B.with_values(np.abs(B.values)), Ch, np.abs(d))
        tau = TAU[np.dtype(A.values.dtype)]
        assert np.all(np.abs(ga.cpu().numpy().astype(np.float64) - rA) <= tau * sA)
        assert np.all(np.abs(gb.cpu().numpy().astype(np.float64) - rB) <= tau * sB)


@pytest.mark.parametrize("t", [None, INF])
@pytest.mark.parametrize("promote,pct", [(1, 300), (2, 125)])
def test_batched_table_size_and_group_promotion(t, promote, pct):
    """The batched forward and backward with other table sizes and light
    columns moved up the lane-group bins, against the oracle."""
    import torch
    from paper_2303_02471_gb300 import ops
    pairs = synth.batch_pairs(16, seed=9, n_scale=0.05)
    As, Bs = _upload_pairs(pairs)
    cfg = ops.Config(t=t, table_slots_pct=pct, group_promote=promote)
    Cs, plan = ops.spgemm_batched(As, Bs, cfg)
    plan.check()
    rng = np.random.default_rng(2)
    dCs = [torch.as_tensor(rng.standard_normal(C.nnz), device="cuda").to(C.values.dtype) for C in Cs]
    gA, gB = ops.spgemm_batched_backward(plan, As, Bs, Cs, dCs)
    plan.check()
    for (A, B), C, dc, ga, gb in zip(pairs, Cs, dCs, gA, gB):
        assert_matches_oracle(C, A, B)
        Ch = C.to_host()
        d = dc.cpu().numpy()
        rA, rB = oracle.backward(A, B, Ch, d)
        sA, sB = oracle.backward(A.with_values(np.abs(A.values)), B.with_values(np.abs(B.values)), Ch, np.abs(d))
        tau = TAU[np.dtype(A.values.dtype)]
        assert np.all(np.abs(ga.cpu().numpy().astype(np.float64) - rA) <= tau * sA)
        assert np.all(np.abs(gb.cpu().numpy().astype(np.float64) - rB) <= tau * sB)


def test_batched_rejects_bad_input():
    from paper_2303_02471_gb300 import ops
    from paper_2303_02471_gb300._native import SpgError
    pairs = synth.batch_pairs(4, seed=7, n_scale=0.03)
    As, Bs = _upload_pairs(pairs)
    bad = Bs[2].rowidx.clone()
    bad[3] = Bs[2].nrows  # out of range
    Bs[2] = ops.CscMatrix(Bs[2].nrows, Bs[2].ncols, Bs[2].colptr, bad, Bs[2].values)
    with pytest.raises(SpgError) as e:
        ops.spgemm_batched_symbolic(As, Bs)
    assert e.value.name == "SPG_ERR_INVALID"


def test_workload4_full_batch_every_product():
    """The 512-product batch (n_i log-uniform 500..20000, Z_i ~ U{2..40}, half
    float64 and half float32), every product against the oracle: structure
    bit-exact, values within tau * sum|a b| (tau = 1e-12 for the float64
    half, 1e-5 for the float32 half); the total product count against its
    closed form (every column of A_i holds Z_i entries, so Op_j = Z_i^2)."""
    from paper_2303_02471_gb300 import ops
    pairs = synth.batch_pairs(512, seed=0)
    As, Bs = _upload_pairs(pairs)
    Cs, plan = ops.spgemm_batched(As, Bs)
    plan.check()
    want = sum(A.ncols * (A.colptr[1] - A.colptr[0]) ** 2 for A, _ in pairs)
    assert plan.info()["products"] == want
    for i, ((A, B), C) in enumerate(zip(pairs, Cs)):
        assert C.values.dtype == (As[i].values.dtype)
        assert_matches_oracle(C, A, B, nthreads=NCPU)


def test_autotune_chooses_and_caches(tmp_path):
    from paper_2303_02471_gb300 import autotune
    pairs = synth.batch_pairs(16, seed=8, n_scale=0.05)
    As, Bs = _upload_pairs(pairs)
    path = str(tmp_path / "tune.json")
    grid = {"t": [257, None], "hash_cta_max": [2048], "cta_threads": [256, 512]}
    cfg, rep = autotune.tune(As, Bs, grid=grid, repeats=1, cache=path)
    assert len(rep["candidates"]) == 4
    cfg2, rep2 = autotune.tune(As, Bs, grid=grid, repeats=1, cache=path)
    assert rep2["config"] == rep["config"]
    from paper_2303_02471_gb300 import ops
    Cs, plan = ops.spgemm_batched(As, Bs, cfg)
    for (A, B), C in zip(pairs, Cs):
        assert_matches_oracle(C, A, B)
    # second stage: table size and lanes per light column around the best
    grid2 = dict(grid, table_slots_pct=[150, 250], group_promote=[0, 1])
    cfg3, rep3 = autotune.tune(As, Bs, grid=grid2, repeats=1, cache=path, refresh=True)
    assert len(rep3["candidates"]) == 4 + 3
    assert {"table_slots_pct", "group_promote"} <= set(rep3["config"])
    Cs, plan = ops.spgemm_batched(As, Bs, cfg3)
    for (A, B), C in zip(pairs, Cs):
        assert_matches_oracle(C, A, B)


def test_product_autotune_chooses_and_caches(tmp_path):
    """The single-product autotuner times its grid on the product, caches the
    pick per pattern signature, and its configuration gives the oracle's C."""
    from paper_2303_02471_gb300 import autotune, ops
    A = synth.rmat(12, seed=3, col_cap=400)
    dA = upload(A)
    path = str(tmp_path / "tune.json")
    grid = {"t": [65, None], "hash_cta_max": [2048], "cta_threads": [512], "small_accumulator": ["hash", "esc"]}
    cfg, rep = autotune.tune_product(dA, dA, grid=grid, repeats=1, cache=path)
    assert len(rep["candidates"]) == 4 and all(r["error"] is None for r in rep["candidates"])
    cfg2, rep2 = autotune.tune_product(dA, dA, grid=grid, repeats=1, cache=path)
    assert rep2["config"] == rep["config"]
    C, plan = ops.spgemm(dA, dA, cfg)
    plan.check()
    assert_matches_oracle(C, A, A)
    # last stage: the pick timed in the single-pass form too
    cfg3, rep3 = autotune.tune_product(dA, dA, grid=dict(grid, form=["two_pass", "single_pass"]), repeats=1,
                                       cache=path, refresh=True)
    assert len(rep3["candidates"]) == 4 + 1 and rep3["form"] in ("two_pass", "single_pass")
    C, plan = ops.spgemm_single_pass(dA, dA, cfg3)
    plan.check()
    assert_matches_oracle(C, A, A)


def _matrix(rng, nrows, lengths, dtype=np.float64):
    cp = np.concatenate([[0], np.cumsum(lengths)]).astype(np.int64)
    rows = np.concatenate([rng.permutation(nrows)[:n] for n in lengths]).astype(np.int32)
    return synth.CSC(nrows, len(lengths), cp, rows, rng.standard_normal(rows.size).astype(dtype))


@pytest.mark.parametrize("dtype", [np.float64, np.float32])
def test_batched_backward_entry_lengths_per_warp(dtype):
    """Entries at the edges of the warp's split (by the whole warp above 64
    products, by 1 to 32 lanes below) in columns of 1 to 70 entries, enough of
    them that the batch's backward works a column per warp.  The longest sum
    (dA) has 6000 terms: 6000 u = 3.6e-4 in float, 6.7e-13 in double."""
    import torch
    from paper_2303_02471_gb300 import ops
    rng = np.random.default_rng(23)
    n, m, k = 6000, 1037, 70
    za = np.array([[0, 1, 2, 7, 8, 9, 31, 32, 33, 63, 64, 65, 127, 128, 129, 300][i % 16] for i in range(k)])
    A = _matrix(rng, m, za, dtype)
    B = _matrix(rng, k, np.arange(n) % 70 + 1, dtype)
    op = np.add.reduceat(za[B.rowidx], B.colptr[:-1])
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    assert op.max() * 10 * sms <= op.sum()
    dA, dB = upload(A, dtype), upload(B, dtype)
    Cs, plan = ops.spgemm_batched([dA], [dB], ops.Config(t=1))
    dc = torch.as_tensor(rng.standard_normal(Cs[0].nnz).astype(dtype), device="cuda")
    full = ops.spgemm_batched_backward(plan, [dA], [dB], Cs, [dc])
    only_b = ops.spgemm_batched_backward(plan, [dA], [dB], Cs, [dc], need_dA=False)
    only_a = ops.spgemm_batched_backward(plan, [dA], [dB], Cs, [dc], need_dB=False)
    plan.check()
    assert only_b[0] is None and only_a[1] is None
    Ch, d = Cs[0].to_host(), dc.cpu().numpy()
    want = oracle.backward(A, B, Ch, d)
    scale = oracle.backward(A.with_values(np.abs(A.values)), B.with_values(np.abs(B.values)), Ch, np.abs(d))
    tau = 1e-12 if dtype == np.float64 else 6000 * 2.0 ** -24
    for got, r, s in ((full[0][0], want[0], scale[0]), (full[1][0], want[1], scale[1]),
                      (only_a[0][0], want[0], scale[0]), (only_b[1][0], want[1], scale[1])):
        assert np.all(np.abs(got.cpu().numpy().astype(np.float64) - r) <= tau * s)


def test_batched_backward_of_skewed_columns_keeps_pace():
    """Columns of one entry of 4000 products and 19 of 4 against columns of 20
    entries of 204: as many products, and as many adds to each place of dA
    (measured equal within a tenth; one lane walking the long entry took 4.6
    times as long)."""
    import torch
    from paper_2303_02471_gb300 import ops
    rng = np.random.default_rng(1)

    def backward_ms(za):
        A, B = upload(_matrix(rng, 5000, za)), upload(_matrix(rng, 20, np.full(600, 20)))
        As, Bs = [A] * 4, [B] * 4
        Cs, plan = ops.spgemm_batched(As, Bs)
        dCs = [torch.randn(C.nnz, dtype=torch.float64, device="cuda") for C in Cs]
        times = []
        for _ in range(9):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            ops.spgemm_batched_backward(plan, As, Bs, Cs, dCs)
            b.record()
            b.synchronize()
            times.append(a.elapsed_time(b))
        plan.check()
        return sorted(times)[4]

    assert backward_ms(np.array([4000] + [4] * 19)) < 2.5 * backward_ms(np.full(20, 204))


def test_batched_backward_reads_the_operands_it_is_given():
    """The same patterns in other buffers than the forward's, whose rows are
    overwritten meanwhile: nothing of the forward's operands is read."""
    import torch
    from paper_2303_02471_gb300 import ops
    pairs = synth.batch_pairs(6, seed=9, n_scale=0.05)
    As, Bs = _upload_pairs(pairs)
    Cs, plan = ops.spgemm_batched(As, Bs)
    dCs = [torch.randn(C.nnz, dtype=C.values.dtype, device="cuda") for C in Cs]
    want = ops.spgemm_batched_backward(plan, As, Bs, Cs, dCs)

    def copy(M):
        return ops.CscMatrix(M.nrows, M.ncols, M.colptr.clone(), M.rowidx.clone(), M.values.clone())
    As2, Bs2 = [copy(M) for M in As], [copy(M) for M in Bs]
    for M in As + Bs:
        M.rowidx.zero_()
    got = ops.spgemm_batched_backward(plan, As2, Bs2, Cs, dCs)
    plan.check()
    for g, w in zip(got[0] + got[1], want[0] + want[1]):
        # sums of at most 1600 terms in another order, in scale with the largest
        tau = 1600 * torch.finfo(w.dtype).eps
        assert (g - w).abs().max() <= tau * 40 * w.abs().max()


def test_batched_plan_refuses_operands_of_other_sizes():
    """Numeric and backward compare the operands' entries with the plan's, as
    the single product does: the gradients are zeroed by the plan's counts."""
    import torch
    from paper_2303_02471_gb300 import ops
    pairs = synth.batch_pairs(4, seed=2, n_scale=0.05)
    As, Bs = _upload_pairs(pairs)
    Cs, plan = ops.spgemm_batched(As, Bs)
    dCs = [torch.ones_like(C.values) for C in Cs]

    def shorter(M):  # one entry less in the last column
        cp = M.colptr.clone()
        cp[-1] -= 1
        return ops.CscMatrix(M.nrows, M.ncols, cp, M.rowidx[:-1].clone(), M.values[:-1].clone())
    for a, b in (([shorter(As[0])] + As[1:], Bs), (As, Bs[:-1] + [shorter(Bs[-1])])):
        with pytest.raises(RuntimeError, match="SPG_ERR_INVALID"):
            ops.spgemm_batched_numeric(plan, a, b)
        with pytest.raises(RuntimeError, match="SPG_ERR_INVALID"):
            ops.spgemm_batched_backward(plan, a, b, Cs, dCs)
    for (A, B), C in zip(pairs, ops.spgemm_batched_numeric(plan, As, Bs)):
        assert_matches_oracle(C, A, B)
    plan.check()
