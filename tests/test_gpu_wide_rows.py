"""CRS_L1 on rows of eight and more entries on average (k_crs_wide: aligned groups
of four entries, realigned in registers; blocks of two and four columns from
sixteen on).  The order of a row's sum is the thread-per-row one, so the product
equals CRS_STAGED's, which walks rows of up to 64 entries the same way, bit for bit."""
import numpy as np
import pytest

import gen
from gpu_util import assert_close, run

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("fp32", [False, True])
@pytest.mark.parametrize("lo,hi", [(8, 8), (9, 9), (16, 16), (27, 27), (0, 64), (33, 63)])
def test_equals_the_staged_product(lib, lo, hi, fp32):
    for n in (1, 2, 3, 255, 256, 257, 1003):     # every phase of the first and last group, and CTA edges
        lens = np.random.default_rng(n).integers(lo, hi + 1, n)
        lens[0] = hi
        A = gen.csr_from_lengths(lens, 300, seed=n)
        for k in (1, 2, 4):
            B = gen.rhs_block(A.n_cols, k, seed=k)
            B = B[:, 0].copy() if k == 1 else B
            with lib.Plan.from_csr(A, variant=lib.SPMV_CRS_L1, val_fp32=fp32) as p, \
                    lib.Plan.from_csr(A, variant=lib.SPMV_CRS_STAGED, val_fp32=fp32) as q:
                y = run(p, B)
                assert np.array_equal(y, run(q, B)), (n, k)
            assert_close(y, A, B, f32val=fp32)


def test_infinities_stay_in_their_rows(lib):
    """A group of four holds entries of the neighbouring rows: their gathers must not reach this row's sum."""
    n, L = 300, 9
    rng = np.random.default_rng(1)
    A = gen.CSR(n, n * L, np.arange(0, n * L + 1, L, dtype=np.int32), np.arange(n * L, dtype=np.int32),
                rng.uniform(-1, 1, n * L))
    B = rng.uniform(-1, 1, n * L)
    B[::2 * L] = np.inf                           # the first entry of every other row
    with lib.Plan.from_csr(A, variant=lib.SPMV_CRS_L1) as p:
        y = run(p, B)
    assert not np.isfinite(y[::2]).any() and np.isfinite(y[1::2]).all()
