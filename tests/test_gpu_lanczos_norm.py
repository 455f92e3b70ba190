"""Lanczos coefficients do not depend on the norm of the start vector: a start block scaled by powers of two,
up to the sizes whose squared norms are still normal numbers, gives the bits of the unscaled one, and every
beta (the last one, which a kernel of its own stores, too) is the oracle's."""
import numpy as np
import pytest

import gen
from oracle import solvers as osol
from gpu_util import dev

pytestmark = pytest.mark.gpu


def scaled(A, f):
    return gen.CSR(A.n_rows, A.n_cols, A.row_ptr, A.col_idx, A.val * f)


@pytest.mark.parametrize("k", [1, 2, 3, 4, 8, 13, 16])
@pytest.mark.parametrize("size", [2.0 ** 60, 1.0, 2.0 ** -60])        # of the matrix: beta_1 is of this size
def test_scaled_start_vectors(lib, k, size):
    A = scaled(gen.eigen_shaped(3001, window=1 << 9), size)
    V0 = gen.rhs_block(A.n_cols, k, seed=k)
    with lib.Plan.from_csr(A) as p, lib.Solver(p, k) as s:
        for m in (1, 2, 6):
            a, b = s.lanczos(dev(V0), m)
            ao, bo = osol.lanczos(A, V0, m)
            # six steps without reorthogonalisation: rounding has not been amplified yet
            assert np.abs(a - ao).max() <= 1e-11 * np.abs(ao).max()
            assert np.abs(b - bo).max() <= 1e-11 * np.abs(bo).max()
            for e in (-480, -200, 3, 500):
                a2, b2 = s.lanczos(dev(V0 * 2.0 ** e), m)
                assert np.array_equal(a2, a) and np.array_equal(b2, b), e


def test_products_of_extreme_start_and_matrix(lib):
    A0 = gen.laplace2d(20)
    V0 = gen.rhs_block(A0.n_cols, 4, seed=2)
    want = None
    for ea, ev in ((0, 0), (500, 505), (-480, -480), (500, -480), (-480, 500)):
        A = scaled(A0, 2.0 ** ea)
        with lib.Plan.from_csr(A) as p, lib.Solver(p, 4) as s:
            a, b = s.lanczos(dev(V0 * 2.0 ** ev), 4)
        a, b = a * 2.0 ** -ea, b * 2.0 ** -ea
        if want is None:
            want = a, b
        assert np.array_equal(a, want[0]) and np.array_equal(b, want[1]), (ea, ev)


def test_product_of_a_large_start_and_a_large_matrix(lib):
    """2^600 I: A V0 overflows for |V0| of 2^480 and more, alpha_1 = 2^600 and beta_1 = 0 do not."""
    n = 700
    A = gen.CSR(n, n, np.arange(n + 1, dtype=np.int32), np.arange(n, dtype=np.int32), np.full(n, 2.0 ** 600))
    for k in (1, 3, 4):
        V0 = np.ones((n, k)) * 2.0 ** 480
        with lib.Plan.from_csr(A) as p, lib.Solver(p, k) as s:
            a, b = s.lanczos(dev(V0), 2)
        assert np.all(a == [[2.0 ** 600], [0.0]]) and not b.any()


def test_columns_of_different_size_and_none(lib):
    """Scales are the column's own; a zero column and one that is not a number give zeros, as before."""
    A = gen.laplace2d(20)
    V0 = gen.rhs_block(A.n_cols, 5, seed=3)
    V0[:, 1] = 0.0
    f = np.array([2.0 ** 400, 1.0, 1.0, 2.0 ** -450, 1.0])
    V1 = V0 * f
    V1[7, 4] = np.nan
    with lib.Plan.from_csr(A) as p, lib.Solver(p, 5) as s:
        a, b = s.lanczos(dev(V0), 5)
        a1, b1 = s.lanczos(dev(V1), 5)
    for c in (0, 2, 3):
        assert np.array_equal(a1[:, c], a[:, c]) and np.array_equal(b1[:, c], b[:, c])
    assert not a1[:, [1, 4]].any() and not b1[:, [1, 4]].any()
