"""An autotune without a candidate that can be built leaves the plan on the kernel it had: AUTO's form of
CRS_L1 (long rows on warps and CTAs), an explicit CRS_L1 (every row on one lane), SELL."""
import numpy as np
import pytest

import gen
from gpu_util import dev, run

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("variant,sigma", [("SPMV_VARIANT_AUTO", 1), ("SPMV_CRS_L1", 1), ("SPMV_SELL", 64)])
def test_failed_autotune_keeps_the_kernel(lib, variant, sigma):
    import torch
    A = gen.powerlaw(20_000, seed=8)            # unsymmetric: SYM cannot be built
    B = gen.uniform(A.n_cols, seed=8)
    C = torch.empty(A.n_rows, dtype=torch.float64, device="cuda")
    with lib.Plan.from_csr(A, variant=getattr(lib, variant), sell_sigma=sigma) as p:
        v0, y0 = p.info().variant, run(p, B)
        for _ in range(2):
            with pytest.raises(lib.SpmvError) as e:
                p.autotune(dev(B), C, [(lib.SPMV_SYM, 1)], reps=2)
            assert e.value.status == 6
            assert p.info().variant == v0 and np.array_equal(run(p, B), y0)
    with lib.Plan.from_csr(A) as p, lib.Plan.from_csr(A, variant=lib.SPMV_CRS_L1) as q:
        assert p.info().variant == q.info().variant and not np.array_equal(run(p, B), run(q, B))
