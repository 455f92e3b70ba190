"""Calls without a stream run on PyTorch's current stream, as it is at the call."""
import numpy as np
import pytest

import gen

pytestmark = pytest.mark.gpu


def test_follows_the_current_stream(lib):
    import threading

    import torch
    from paper_1101_0091_gb300._binding import current_stream
    assert current_stream() == torch.cuda.current_stream().cuda_stream
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        assert current_stream() == s.cuda_stream
    seen = []
    t = threading.Thread(target=lambda: seen.append(current_stream()))   # another thread has its own
    with torch.cuda.stream(s):
        t.start()
        t.join()
    assert seen == [torch.cuda.default_stream().cuda_stream] and current_stream() != s.cuda_stream
    A = gen.poisson3d_var(20)
    B = torch.from_numpy(gen.uniform(A.n_cols, seed=1)).cuda()
    C, D = torch.zeros_like(B), torch.zeros_like(B)
    with lib.Plan.from_csr(A) as p:
        p.apply(B, D)
        torch.cuda.synchronize()
        s.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(s):
            torch.cuda._sleep(20_000_000)      # the product is behind this on s
            p.apply(B, C)
            done = torch.cuda.Event()
            done.record()
        assert not done.query()
        done.synchronize()
        assert np.array_equal(C.cpu().numpy(), D.cpu().numpy())
