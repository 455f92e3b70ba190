"""Widths of the batch kernels' accesses to B and C (1, 2 or 4 doubles, by k, row strides and
addresses): the same bits on every width, nothing written beside the rows' k values."""
import numpy as np
import pytest

import gen
import oracle
from gpu_util import TOL_FP64, dev, host

pytestmark = pytest.mark.gpu


def placed(n, k, ld, off, block=None):
    """n x k block with row stride ld that starts off doubles past a 256-byte boundary, and its buffer."""
    import torch
    buf = torch.full((off + n * ld + 8,), -7.0, dtype=torch.float64, device="cuda")
    view = buf[off:off + n * ld].view(n, ld)[:, :k]
    if block is not None:
        view.copy_(dev(block))
    return buf, view


@pytest.mark.parametrize("k", [1, 2, 3, 4, 6, 8, 12, 16])
@pytest.mark.parametrize("policy", ["SPMV_BATCH_SORTED", "SPMV_BATCH_ADAPT", "SPMV_BATCH_L4", "noalloc"])
def test_same_bits(lib, k, policy):
    import torch
    lens = np.concatenate([np.arange(0, 70), np.full(200, 1), np.full(100, 2), np.full(70, 3), np.full(40, 4), [300]])
    As = [gen.csr_from_lengths(np.random.default_rng(m).permutation(lens), 333, seed=m) for m in range(3)]
    Bs = [gen.rhs_block(333, k, seed=m) for m in range(3)]
    plans = [lib.Plan.from_csr(A) for A in As]
    dA = [tuple(dev(x) for x in (A.row_ptr, A.col_idx, A.val)) for A in As]
    ref = None
    for ld, off in ((k, 0), (k, 1), (k, 2), (k, 4), (k + 1, 0), (k + 2, 0), (k + 4, 0)):
        Bd = [placed(A.n_cols, k, ld, off, B) for A, B in zip(As, Bs)]
        Cd = [placed(A.n_rows, k, ld, off) for A in As]
        if policy == "noalloc":
            p = lambda ts: [t.data_ptr() for t in ts]
            lib.spmv_batch_apply_noalloc([A.n_rows for A in As], *(p([d[i] for d in dA]) for i in range(3)),
                                         p([v for _, v in Bd]), [ld] * 3, p([v for _, v in Cd]), [ld] * 3, k)
        else:
            with lib.Batch(plans, k, [getattr(lib, policy)] * 3) as b:
                b.set_io([v for _, v in Bd], [v for _, v in Cd])
                b.apply()
                torch.cuda.synchronize()
        ys = [host(v).copy() for _, v in Cd]
        for (buf, v) in Cd:
            v.fill_(-7.0)
            assert (host(buf) == -7.0).all()
        ref = ref or ys
        for A, B, y, r in zip(As, Bs, ys, ref):
            assert np.array_equal(y, r), (ld, off)
    for A, B, y in zip(As, Bs, ref):
        assert oracle.max_err_ratio(y, oracle.spmm(A, B), oracle.abs_scale(A, B), TOL_FP64) <= 1.0
    for p in plans:
        p.close()
