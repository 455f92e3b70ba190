"""SELL blocks at the sizes where the columns per lane change (four, two and one; 16- and 8-byte accesses):
the bits of an explicit CRS_L1 product, which sums a row in the same order, and the oracle's values."""
import numpy as np
import pytest

import gen
from gpu_util import assert_close, dev, host

pytestmark = pytest.mark.gpu


def quick(n, lo, hi, seed):
    """Rows of lo .. hi entries, random columns (repeats allowed)."""
    rng = np.random.default_rng(seed)
    lens = rng.integers(lo, hi + 1, n)
    rp = np.zeros(n + 1, np.int32)
    rp[1:] = np.cumsum(lens)
    return gen.CSR(n, n, rp, rng.integers(0, n, rp[-1]).astype(np.int32), rng.uniform(-1, 1, rp[-1]))


# rows, lengths, k: four columns (k = 16, 12, 4), two (8 at 100,003; 2; 6), their neighbours with one
@pytest.mark.parametrize("n,lo,hi,k", [(250_001, 0, 7, 16), (249_999, 0, 7, 16), (333_334, 1, 3, 12), (1_000_000, 0, 3, 4),
                                       (100_003, 0, 12, 8), (100_003, 10, 20, 16), (200_001, 0, 2, 2), (199_999, 0, 3, 2),
                                       (400_001, 1, 3, 2), (400_001, 4, 6, 2), (133_337, 2, 5, 6)])
@pytest.mark.parametrize("fp32", [False, True])
def test_widths(lib, n, lo, hi, k, fp32):
    import torch
    A = quick(n, lo, hi, seed=k)
    B = gen.rhs_block(n, k, seed=k)
    with lib.Plan.from_csr(A, val_fp32=fp32, variant=lib.SPMV_SELL, sell_sigma=256) as p:
        ys = []
        for ld, off in ((k, 0), (k + 1, 0), (k, 1), (k + 2, 0)):
            Bd = torch.full((n * ld + off,), 7.0, dtype=torch.float64, device="cuda")[off:].view(-1, ld)
            C = torch.full((n * ld + off,), 7.0, dtype=torch.float64, device="cuda")[off:].view(-1, ld)
            Bd[:, :k] = dev(B)
            p.apply_block(Bd, C, k)
            y = host(C)
            assert np.all(y[:, k:] == 7.0)
            ys.append(np.ascontiguousarray(y[:, :k]))
        p.set_variant(lib.SPMV_CRS_L1)
        C = torch.empty((n, k), dtype=torch.float64, device="cuda")
        p.apply_block(dev(B), C, k)
        want = host(C)
    for y in ys:
        assert np.array_equal(y, want)
    assert_close(want, A, B, f32val=fp32)


@pytest.mark.parametrize("longest", [64, 65, 300])
@pytest.mark.parametrize("fp32", [False, True])
def test_one_long_row(lib, longest, fp32):
    """Two columns per lane in unrolled slots from a row of more than 64 entries on."""
    A = quick(200_001, 1, 3, seed=longest)
    lens = np.diff(A.row_ptr)
    lens[77_777] = longest
    rp = np.zeros(A.n_rows + 1, np.int32)
    rp[1:] = np.cumsum(lens)
    rng = np.random.default_rng(longest)
    A = gen.CSR(A.n_rows, A.n_cols, rp, rng.integers(0, A.n_cols, rp[-1]).astype(np.int32), rng.uniform(-1, 1, rp[-1]))
    import torch
    for k, ld in ((2, 2), (4, 4), (4, 5), (6, 6)):
        B = gen.rhs_block(A.n_cols, k, seed=k)
        Bd = torch.full((A.n_cols, ld), 7.0, dtype=torch.float64, device="cuda")
        Bd[:, :k] = dev(B)
        got = []
        for variant in (lib.SPMV_SELL, lib.SPMV_CRS_L1):
            with lib.Plan.from_csr(A, val_fp32=fp32, variant=variant, sell_sigma=256) as p:
                C = torch.full((A.n_rows, ld), 7.0, dtype=torch.float64, device="cuda")
                p.apply_block(Bd, C, k)
                got.append(host(C))
        assert np.array_equal(got[0], got[1]) and np.all(got[0][:, k:] == 7.0)
        assert_close(np.ascontiguousarray(got[0][:, :k]), A, B, f32val=fp32)
