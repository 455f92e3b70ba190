"""The solvers' vector kernels at the edges of their walks: blocks whose units end
inside a CTA, a pair or a step, every way of walking (pairs, rows, column groups,
and the flat walk of the other k), one CTA and several, against the oracle."""
import numpy as np
import pytest

import gen
from oracle import solvers as osol
from gpu_util import dev, host

pytestmark = pytest.mark.gpu


def spd(n):
    """Tridiagonal, diagonally dominant."""
    rng = np.random.default_rng(n)
    off = -rng.uniform(0.5, 1.0, max(n - 1, 0))
    d = np.full(n, 2.5)
    rows = np.concatenate([np.arange(n), np.arange(n - 1), np.arange(1, n)])
    cols = np.concatenate([np.arange(n), np.arange(1, n), np.arange(n - 1)])
    vals = np.concatenate([d, off, off])
    order = np.lexsort((cols, rows))
    rp = np.zeros(n + 1, np.int32)
    rp[1:] = np.cumsum(np.bincount(rows, minlength=n))
    return gen.CSR(n, n, rp, cols[order].astype(np.int32), vals[order])


def rel(a, b):
    return np.linalg.norm(a - b) / max(np.linalg.norm(b), 1e-300)


@pytest.mark.parametrize("k", [1, 2, 3, 4, 5, 7, 8, 9, 11, 12, 15, 16])
@pytest.mark.parametrize("n", [1, 2, 3, 170, 511, 1023, 1025, 40_001])
def test_cg_and_lanczos_match_oracle(lib, n, k):
    A = spd(n)
    B = gen.rhs_block(n, k, seed=k)
    steps = min(n, 4)
    with lib.Plan.from_csr(A) as p, lib.Solver(p, k) as s:
        X = dev(np.zeros((n, k)))
        it, rr, _ = s.cg(dev(B), X, max_iter=steps, rtol=0.0, check_every=3)
        X = host(X)
        Xo, info = osol.cg(A, B, max_iter=steps, rtol=0.0)
        if n > 4:      # at n <= 4 the last residual is rounding alone
            assert np.all(it == steps)
            assert np.all(np.abs(rr - info["rr"]) <= 1e-8 * info["rr"])
        for c in range(k):
            assert rel(X[:, c], Xo[:, c]) < 1e-10
        m = min(n, 3)
        a, b = s.lanczos(dev(B), m)
        ao, bo = osol.lanczos(A, B, m)[:2]
        assert np.abs(a - ao).max() <= 1e-11 * np.abs(ao).max()
        assert np.abs(b[:m - 1] - bo[:m - 1]).max(initial=0.0) <= 1e-11 * np.abs(ao).max()
