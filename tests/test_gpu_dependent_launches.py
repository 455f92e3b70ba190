"""Products launched one behind the other on a stream may start while the last CTAs
of the kernel before still run, and wait for it before they touch B or C: chains in
which every product reads what the one before wrote (and overwrites what the one
before read) equal the same chain with a synchronisation after every call, bit for
bit, for every kernel that is launched that way, between foreign kernels and from a
captured graph."""
import numpy as np
import pytest

import gen
from gpu_util import dev, host

pytestmark = pytest.mark.gpu


def forms(lib):
    short = gen.poisson3d_var(30, seed=1)
    wide = gen.csr_from_lengths(np.full(6000, 20), 6000, seed=2)
    lens = np.random.default_rng(3).integers(1, 6, 9000)
    lens[::900] = 700
    long_rows = gen.csr_from_lengths(lens, 9000, seed=3)
    eigen = gen.eigen_shaped(30_000, window=1 << 12)
    return {"row": (short, lib.SPMV_CRS_L1, (1, 2, 3, 8)), "wide": (wide, lib.SPMV_CRS_L1, (1, 2, 4)),
            "long": (long_rows, lib.SPMV_VARIANT_AUTO, (1, 2, 4, 5)), "sell": (eigen, lib.SPMV_SELL, (1, 3, 4)),
            "lanes": (short, lib.SPMV_CRS_L4, (1, 4)), "staged": (short, lib.SPMV_CRS_STAGED, (1, 4))}


def chain(plan, x0, steps, between, sync):
    import torch
    x, y = dev(x0), torch.empty(x0.shape, dtype=torch.float64, device="cuda")
    for i in range(steps):
        plan.apply_block(x, y, x0.shape[1])
        if sync:
            torch.cuda.synchronize()
        if between and i % 3 == 2:      # a foreign kernel that reads the result and writes the next operand
            torch.mul(y, 1.0 / 16, out=y)
        x, y = y, x
    return host(x)


@pytest.mark.parametrize("name", ["row", "wide", "long", "sell", "lanes", "staged"])
def test_chains_equal_synchronised_chains(lib, name):
    import torch
    A, variant, ks = forms(lib)[name]
    A.val = A.val / 8
    with lib.Plan.from_csr(A, variant=variant, sell_sigma=64) as p:
        for k in ks:
            x0 = gen.rhs_block(A.n_cols, k, seed=k)
            for between in (False, True):
                want = chain(p, x0, 40, between, True)
                assert np.isfinite(want).all()
                for _ in range(3):
                    assert np.array_equal(chain(p, x0, 40, between, False), want), (k, between)
            # the same chain (an even number of steps, so that it ends where it began) from a graph
            x, y = dev(x0), torch.zeros(x0.shape, dtype=torch.float64, device="cuda")
            s = torch.cuda.Stream()
            with torch.cuda.stream(s):
                p.apply_block(x, y, k)
            torch.cuda.synchronize()
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g, stream=s):
                for _ in range(10):
                    p.apply_block(x, y, k)
                    p.apply_block(y, x, k)
            x.copy_(dev(x0))
            g.replay()
            g.replay()
            torch.cuda.synchronize()
            assert np.array_equal(host(x), chain(p, x0, 40, False, True))


def test_split_chain_equals_the_synchronised_one(lib):
    """The halo pass and the next local pass start behind one another the same way."""
    import torch
    A = gen.poisson3d_var(40)
    h = A.n_cols - A.n_cols // 10
    x0 = gen.uniform(A.n_cols, seed=3)
    halo = torch.from_numpy(x0[h:].copy()).pin_memory()
    copy = torch.cuda.Stream()
    with lib.Plan.from_csr(A, halo_begin=h) as p:
        got = []
        for sync in (True, False, False):
            B, C = dev(x0.copy()), torch.zeros(A.n_rows, dtype=torch.float64, device="cuda")
            for _ in range(20):
                p.apply_split(B, halo, C, copy_stream=copy)
                if sync:
                    torch.cuda.synchronize()
                torch.mul(C[:h], 1.0 / 32, out=B[:h])
                p.apply_split(B, halo, C, copy_stream=copy)
                if sync:
                    torch.cuda.synchronize()
            got.append(host(C))
        assert np.isfinite(got[0]).all() and all(np.array_equal(g, got[0]) for g in got)
