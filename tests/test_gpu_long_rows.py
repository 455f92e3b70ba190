"""AUTO's CRS_L1 on matrices whose few long rows take a warp or a CTA each
(k_crs_long): row lengths at the edges of the three row classes, every block
width and alignment, against the oracle; the choice of the form; values that
masked lanes must not touch."""
import numpy as np
import pytest

import gen
import oracle
from gpu_util import assert_close, dev, host, run

pytestmark = pytest.mark.gpu

EDGES = [0, 1, 31, 32, 33, 48, 49, 63, 64, 65, 127, 129, 511, 512, 513, 1023, 2047, 4097]


def matrix(seed, integer=False, n_cols=5000):
    """1200 short rows with the edge lengths spread between them (1.5 % long rows)."""
    lens = np.random.default_rng(seed).integers(0, 9, 1200)
    lens[np.arange(len(EDGES)) * 64 + 5] = EDGES
    return gen.csr_from_lengths(lens, n_cols, seed, integer=integer)


@pytest.mark.parametrize("k", [1, 2, 3, 4, 6, 7, 8, 13, 16])
@pytest.mark.parametrize("fp32", [False, True])
def test_edges_match_oracle_whatever_the_layout(lib, k, fp32):
    import torch
    A = matrix(3)
    B = gen.rhs_block(A.n_cols, k, seed=k)
    with lib.Plan.from_csr(A, val_fp32=fp32) as p:
        y0 = None
        for ldb, ldc, off in ((k, k, 0), (k + 1, k, 0), (k + 2, k + 3, 0), (k, k, 1)):
            Bd = torch.full((A.n_cols * ldb + off,), 7.0, dtype=torch.float64, device="cuda")[off:].view(-1, ldb)
            C = torch.full((A.n_rows * ldc + off,), 7.0, dtype=torch.float64, device="cuda")[off:].view(-1, ldc)
            Bd[:, :k] = dev(B)
            p.apply_block(Bd, C, k)
            y = host(C)
            assert np.all(y[:, k:] == 7.0)
            y = np.ascontiguousarray(y[:, :k])
            if y0 is None:
                y0 = y
            assert np.array_equal(y, y0)        # the order of a row's sum does not depend on the layout
    assert_close(y0, A, B, f32val=fp32)


def test_integer_exact_and_chosen_by_auto_only(lib):
    A = matrix(4, integer=True)
    B = np.random.default_rng(1).integers(-1024, 1025, A.n_cols).astype(np.float64)
    U = gen.uniform(A.n_cols, seed=2)
    with lib.Plan.from_csr(A) as p, lib.Plan.from_csr(A, variant=lib.SPMV_CRS_L1) as q:
        assert p.info().variant == q.info().variant == lib.SPMV_CRS_L1
        assert_close(run(p, B), A, B, exact=True)
        y_auto, y_l1 = run(p, U), run(q, U)
        q.set_variant(lib.SPMV_VARIANT_AUTO)    # the same form as a plan created with AUTO
        assert np.array_equal(run(q, U), y_auto)
        p.set_variant(lib.SPMV_CRS_L1)          # an explicit CRS_L1 keeps a row on one lane
        assert np.array_equal(run(p, U), y_l1)


def test_only_long_rows_and_one_dense_row(lib):
    for lens in ([4097], [200] + [0] * 9, [3000] * 3 + [2] * 30):
        A = gen.csr_from_lengths(lens, 5000, seed=6)
        B = gen.rhs_block(A.n_cols, 3, seed=6)
        with lib.Plan.from_csr(A) as p:
            assert_close(run(p, B[:, 0].copy()), A, B[:, 0].copy())
            assert_close(run(p, B), A, B)


def test_infinities_stay_in_their_rows(lib):
    A = matrix(5, n_cols=20000)
    bad = int(A.col_idx[A.row_ptr[5 + 64 * 12]])            # a column of one long row
    hit = np.zeros(A.n_rows, bool)
    hit[np.repeat(np.arange(A.n_rows), np.diff(A.row_ptr))[A.col_idx == bad]] = True
    B = gen.rhs_block(A.n_cols, 4, seed=8)
    with lib.Plan.from_csr(A) as p:
        for k in (1, 4):
            Bk = B[:, 0].copy() if k == 1 else B
            y = run(p, Bk)
            Bi = Bk.copy()
            Bi[bad] = np.inf
            yi = run(p, Bi)
            assert np.array_equal(yi[~hit], y[~hit]) and not np.isfinite(yi[hit]).any()
    assert hit.any() and oracle.spmv(A, B[:, 0].copy()).shape == (A.n_rows,)


def quick(lens, n_cols, seed):
    """Rows of the given lengths, random columns (repeats allowed)."""
    rng = np.random.default_rng(seed)
    rp = np.zeros(len(lens) + 1, np.int32)
    rp[1:] = np.cumsum(lens)
    return gen.CSR(len(lens), n_cols, rp, rng.integers(0, n_cols, rp[-1]).astype(np.int32),
                   rng.uniform(-1, 1, rp[-1]))


@pytest.mark.parametrize("k", [1, 3, 8, 16])
def test_classes_of_rows(lib, k):
    """Where a lane's rows end (12 entries, or 32 when a quarter of the rows exceed 12), where a warp's end
    for this k, and more than 16,384 long rows (warps up to 512 entries)."""
    rng = np.random.default_rng(k)
    few = rng.integers(0, 13, 3000)
    few[::60] = rng.choice([11, 12, 13, 14, 32 + 512 // k, 33 + 512 // k, 700], 50)
    half = np.where(rng.random(3000) < 0.5, rng.integers(13, 33, 3000), 3)
    half[::200] = [33, 34, 60, 64, 100, 500, 544, 545, 600, 1000, 31, 32, 33, 70, 90]
    many = np.full(80_000, 2)
    many[::4] = rng.integers(13, 60, 20_000)
    many[1] = 900
    for lens in (few, half, many):
        A = quick(lens, 4000, seed=k)
        B = gen.rhs_block(A.n_cols, k, seed=k)
        B = B[:, 0].copy() if k == 1 else B
        with lib.Plan.from_csr(A) as p:
            assert p.info().variant == lib.SPMV_CRS_L1
            assert_close(run(p, B), A, B)
