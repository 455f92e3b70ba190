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


def big(n, lo, hi, seed):
    """n rows of lo .. hi entries (columns may repeat)."""
    rng = np.random.default_rng(seed)
    lens = rng.integers(lo, hi + 1, n)
    rp = np.zeros(n + 1, np.int32)
    rp[1:] = np.cumsum(lens)
    return gen.CSR(n, 5000, rp, rng.integers(0, 5000, rp[-1]).astype(np.int32), rng.uniform(-1, 1, rp[-1]))


@pytest.mark.parametrize("vname,fp32", [("SPMV_CRS_L1", False), ("SPMV_CRS_L1", True), ("SPMV_SELL", False)])
@pytest.mark.parametrize("lo,hi", [(3, 3), (0, 5), (17, 17)])
def test_several_columns_per_lane_equal_the_vector_product(lib, lo, hi, vname, fp32):
    """Enough rows for two to seven columns per lane: even rows (up to four), uneven ones (two), longer
    ones (no 3, 5, 7 in CRS_L1), in aligned and unaligned blocks."""
    A = big(400_013 if hi < 16 else 60_001, lo, hi, seed=hi)
    with lib.Plan.from_csr(A, variant=getattr(lib, vname), sell_sigma=64, val_fp32=fp32) as p:
        B = gen.rhs_block(A.n_cols, 16, seed=1)
        want = np.empty((A.n_rows, 16))
        for c in range(16):
            y = block(A.n_rows, 1, 0)
            p.apply(dev(B[:, c]), y)
            want[:, c] = host(y)[:, 0]
        for k in (2, 3, 4, 5, 6, 7, 8, 9, 10, 14, 15, 16):
            for ld, off in ((k, 0), (k + 1, 0), (k, 1)):
                Bd, C = block(A.n_cols, ld, off), block(A.n_rows, ld, off)
                Bd[:, :k] = dev(B[:, :k])
                p.apply_block(Bd, C, k)
                y = host(C)
                assert np.array_equal(y[:, :k], want[:, :k]), (k, ld, off)
                assert np.all(y[:, k:] == 7.0)
