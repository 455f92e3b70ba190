"""Blocks of every k through the column-split kernels (k_crs_cols, k_sell_cols):
odd k, odd leading dimensions and blocks 8 bytes off take one column per lane,
even aligned ones two or four.  A column's entries are summed in the order of the
single-vector kernel, so each column equals that product bit for bit, and the
columns beyond k are not written."""
import numpy as np
import pytest

import gen
from gpu_util import assert_close, dev, host

pytestmark = pytest.mark.gpu


def block(n, ld, off):
    import torch
    return torch.full((n * ld + off,), 7.0, dtype=torch.float64, device="cuda")[off:].view(n, ld)


@pytest.mark.parametrize("k", [2, 3, 4, 5, 6, 7, 9, 10, 12, 13, 15, 16])
@pytest.mark.parametrize("vname,fp32", [("SPMV_CRS_L1", False), ("SPMV_CRS_L1", True), ("SPMV_SELL", False),
                                        ("SPMV_SELL", True)])
def test_every_column_equals_the_vector_product(lib, k, vname, fp32):
    rows_per_cta = 256 // k                     # one column per lane
    sizes = [1, rows_per_cta - 1, rows_per_cta, rows_per_cta + 1, 777]
    mats = [gen.csr_from_lengths(np.random.default_rng(n).integers(0, 12, n), 900, seed=n) for n in sizes]
    mats.append(gen.powerlaw(1500, seed=3, lmax=300))
    for A in mats:
        B = gen.rhs_block(A.n_cols, k, seed=k)
        with lib.Plan.from_csr(A, variant=getattr(lib, vname), sell_sigma=64, val_fp32=fp32) as p:
            want = np.empty((A.n_rows, k))
            for c in range(k):
                y = block(A.n_rows, 1, 0)
                p.apply(dev(B[:, c]), y)
                want[:, c] = host(y)[:, 0]
            for ldb, ldc, off in ((k, k, 0), (k + 1, k, 0), (k + 2, k + 3, 0), (k, k, 1), (k + 2, k + 2, 1)):
                Bd, C = block(A.n_cols, ldb, off), block(A.n_rows, ldc, off)
                Bd[:, :k] = dev(B)
                p.apply_block(Bd, C, k)
                y = host(C)
                assert np.array_equal(y[:, :k], want), (ldb, ldc, off)
                assert np.all(y[:, k:] == 7.0)
        assert_close(want, A, B, f32val=fp32)
