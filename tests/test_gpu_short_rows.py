"""CRS_L1 on short rows, one vector (k_crs_row: four entries at a time, then the
last 0..3): every row length modulo four, alone and mixed in a warp, unit and
strided vectors, against CRS_STAGED's product (the same order of the sums)."""
import numpy as np
import pytest

import gen
from gpu_util import assert_close, dev, host, run

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("fp32", [False, True])
@pytest.mark.parametrize("lo,hi", [(0, 0), (1, 1), (2, 2), (3, 3), (4, 4), (5, 5), (6, 6), (7, 7), (0, 7), (0, 15)])
def test_equals_the_staged_product(lib, lo, hi, fp32):
    for n in (1, 31, 256, 257, 1003):
        lens = np.random.default_rng(n + hi).integers(lo, hi + 1, n)
        A = gen.csr_from_lengths(np.minimum(lens, np.arange(n) % 8 + lo), 60, seed=n)   # below 8 on average
        B = gen.uniform(A.n_cols, seed=3)
        with lib.Plan.from_csr(A, variant=lib.SPMV_CRS_L1, val_fp32=fp32) as p, \
                lib.Plan.from_csr(A, variant=lib.SPMV_CRS_STAGED, val_fp32=fp32) as q:
            y = run(p, B)
            assert np.array_equal(y, run(q, B))
            import torch
            Bs = torch.full((A.n_cols, 3), 7.0, dtype=torch.float64, device="cuda")
            Cs = torch.full((A.n_rows, 2), 7.0, dtype=torch.float64, device="cuda")
            Bs[:, 0] = dev(B)
            p.apply_block(Bs, Cs, 1)              # one column of wider blocks
            c = host(Cs)
            assert np.array_equal(c[:, 0], y) and np.all(c[:, 1] == 7.0)
        assert_close(y, A, B, f32val=fp32)
