"""The ESC accumulator at the edges of its bins, against the oracle."""
import os

import numpy as np
import pytest

import oracle
from paper_2303_02471_gb300 import synth

from gpu_helpers import assert_matches_oracle, upload

pytestmark = pytest.mark.gpu

NCPU = len(os.sched_getaffinity(0))


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


@pytest.mark.parametrize("dtype", [np.float64, np.float32])
@pytest.mark.parametrize("m,empty", [(5000, 0), (5000, 70), (300, 3), (40, 0)])
def test_column_lengths(m, empty, dtype):
    """Columns of exactly op products for op around every bin's limit, with
    `empty` entries of B that meet empty columns of A in front of, between and
    behind the others (more entries than lanes), rows that differ (m = 5000)
    and rows that repeat; alone, in a single pass and counted only."""
    from paper_2303_02471_gb300 import ops
    rng = np.random.default_rng(m + empty)
    ops_of = [0, 1, 2, 7, 8, 9, 15, 16, 17, 31, 32, 33, 63, 64, 65, 127, 128, 129, 255, 256] * 3
    # A's columns: 32 of every length 0..20
    za = np.repeat(np.arange(21), 32)
    A = synth.CSC(m, za.size, np.concatenate([[0], np.cumsum(za)]).astype(np.int64),
                  np.concatenate([rng.permutation(m)[:z] for z in za]).astype(np.int32),
                  rng.standard_normal(za.sum()).astype(dtype))
    cols = []
    for op in ops_of:
        ks, left = [], op
        while left:
            z = int(rng.integers(1, min(20, left) + 1))
            ks.append(z * 32 + int(rng.integers(0, 32)))
            left -= z
        ks += list(rng.integers(0, 32, empty))
        cols.append(rng.permutation(ks).astype(np.int32))
    B = synth.CSC(za.size, len(cols), np.concatenate([[0], np.cumsum([len(c) for c in cols])]).astype(np.int64),
                  np.concatenate(cols).astype(np.int32), rng.standard_normal(sum(len(c) for c in cols)).astype(dtype))
    ref = oracle.spgemm(A, B, nthreads=NCPU)
    dA, dB = upload(A, dtype), upload(B, dtype)
    for cfg in (ops.Config(), ops.Config(small_accumulator="esc"), ops.Config(small_accumulator="esc", group_promote=2)):
        for call in (ops.spgemm, ops.spgemm_single_pass):
            C, plan = call(dA, dB, cfg)
            plan.check()
            assert np.array_equal(plan.op_counts().cpu().numpy(), ops_of)
            assert_matches_oracle(C, A, B, ref=ref)


def test_rows_beyond_32_bit_keys():
    """More than 2^24 numbered rows: (row, place) of the bin of 256 products
    needs 64 bits, that of the smaller bins 32."""
    from paper_2303_02471_gb300 import ops
    rng = np.random.default_rng(3)
    k = 17 << 17
    m = 8 * k
    arow = rng.permutation(m).astype(np.int32).reshape(k, 8)
    arow[1::2, 0] = arow[0::2, 0]  # A's columns 2q and 2q + 1 share a row
    A = synth.CSC(m, k, np.arange(0, m + 1, 8, dtype=np.int64), arow.ravel(), rng.standard_normal(m))
    z = np.repeat([1, 3, 8, 16, 17, 31, 32], 4)
    cols = []
    for n in z:
        r = 2 * rng.choice(k // 2, n, replace=False) + rng.integers(0, 2, n)
        if n >= 2:
            r[1] = r[0] ^ 1
        cols.append(r)
    B = synth.CSC(k, z.size, np.concatenate([[0], np.cumsum(z)]).astype(np.int64),
                  np.concatenate(cols).astype(np.int32), rng.standard_normal(int(z.sum())))
    C, plan = ops.spgemm(upload(A), upload(B), ops.Config(small_accumulator="esc", scratch_cap_bytes=1 << 26))
    plan.check()
    assert_matches_oracle(C, A, B)
