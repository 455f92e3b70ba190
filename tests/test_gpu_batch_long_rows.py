"""Batch members' long rows at k = 2: four entries per lane and round (row classes of
one lane count).  The last round of a row is partly past its end on some lanes."""
import numpy as np
import pytest

import gen
import oracle
from gpu_util import TOL_FP64, dev, host

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("special", [False, True])
@pytest.mark.parametrize("policy", ["SPMV_BATCH_SORTED", "SPMV_BATCH_ADAPT"])
def test_row_ends(lib, policy, special):
    import torch
    As, Bs = [], []
    for m, around in enumerate((33, 64, 65, 128, 256, 512, 1024, 1250)):
        lens = np.clip(np.arange(around - 20, around + 21), 0, 1300)
        As.append(gen.csr_from_lengths(lens, 1301, seed=m))
        Bs.append(gen.rhs_block(1301, 2, seed=m))
        if special:     # an infinity must stay in its rows
            last = As[-1].col_idx[As[-1].row_ptr[1:] - 1]
            Bs[-1][np.setdiff1d(As[-1].col_idx, last)[:1]] = np.inf
    plans = [lib.Plan.from_csr(A) for A in As]
    Bd = [dev(B) for B in Bs]
    Cd = [torch.full((A.n_rows, 2), float("nan"), dtype=torch.float64, device="cuda") for A in As]
    with lib.Batch(plans, 2, [getattr(lib, policy)] * len(As)) as b:
        b.set_io(Bd, Cd)
        b.apply()
        torch.cuda.synchronize()
    for A, B, C in zip(As, Bs, Cd):
        y, ref = host(C), oracle.spmm(A, B)
        ok = np.isfinite(ref).all(1)
        assert np.array_equal(np.isfinite(y), np.isfinite(ref))
        assert special or ok.all()
        scale = oracle.abs_scale(A, np.where(np.isfinite(B), B, 0.0))
        assert oracle.max_err_ratio(y[ok], ref[ok], scale[ok], TOL_FP64) <= 1.0
    for p in plans:
        p.close()
