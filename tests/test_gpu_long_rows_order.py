"""The order of AUTO's long rows (longest first, ties by row) decides which rows take a CTA: lengths on both
sides of the counting sort's last bucket (1023 entries) and of the CTA's threshold, ties, shuffled over the
matrix, against the oracle."""
import numpy as np
import pytest

import gen
from gpu_util import assert_close, run

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k", [1, 2, 16])
def test_lengths_around_the_buckets(lib, k):
    rng = np.random.default_rng(k)
    lens = rng.integers(0, 9, 4000)
    at = rng.permutation(4000)
    edge = [13, 33, 32 + 512 // k, 33 + 512 // k, 512, 513, 544, 545, 1021, 1022, 1023, 1024, 1025, 1500, 3000]
    lens[at[:45]] = edge * 3
    A = gen.csr_from_lengths(lens, 4500, seed=k)
    B = gen.rhs_block(A.n_cols, k, seed=k)
    B = B[:, 0].copy() if k == 1 else B
    with lib.Plan.from_csr(A) as p:
        assert p.info().variant == lib.SPMV_CRS_L1
        y = run(p, B)
        assert_close(y, A, B)
    # the same rows in another order: a row's sum does not depend on where it stands in the list's classes
    perm = rng.permutation(4000)
    rows = [slice(A.row_ptr[i], A.row_ptr[i + 1]) for i in perm]
    rp = np.concatenate([[0], np.cumsum(lens[perm])]).astype(np.int32)
    P = gen.CSR(4000, 4500, rp, np.concatenate([A.col_idx[s] for s in rows]), np.concatenate([A.val[s] for s in rows]))
    with lib.Plan.from_csr(P) as p:
        assert np.array_equal(run(p, B), y[perm])
