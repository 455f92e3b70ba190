"""The local/halo product inside a captured graph: the halo pass is launched dependently behind the local pass
and an event wait (the copy on its own stream), or behind the local pass alone (one stream); replays with new
operands equal the direct call bit for bit."""
import numpy as np
import pytest

import gen
from gpu_util import dev, host

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("two_streams", [False, True])
@pytest.mark.parametrize("fp32", [False, True])
def test_split_in_a_graph(lib, two_streams, fp32):
    import torch
    A = gen.poisson3d_var(24)
    h = A.n_cols - A.n_cols // 8
    s, copy = torch.cuda.Stream(), torch.cuda.Stream()
    halo = torch.zeros(A.n_cols - h, dtype=torch.float64).pin_memory()
    B = torch.zeros(A.n_cols, dtype=torch.float64, device="cuda")
    C = torch.zeros(A.n_rows, dtype=torch.float64, device="cuda")
    with lib.Plan.from_csr(A, halo_begin=h, val_fp32=fp32) as p:
        call = lambda: p.apply_split(B, halo, C, s, copy if two_streams else None)
        torch.cuda.synchronize()
        call()
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            call()
            call()
        for seed in range(3):
            x = gen.uniform(A.n_cols, seed=seed)
            halo.copy_(torch.from_numpy(x[h:]))
            got = []
            for run in (call, g.replay):
                B.copy_(dev(x))
                B[h:] = np.nan
                C.fill_(np.nan)
                torch.cuda.synchronize()
                run()
                got.append(host(C))
            assert np.isfinite(got[0]).all() and np.array_equal(got[0], got[1])
