"""Batched jobs with a scale wider than 256, at batch sizes where the launch
holds more blocks than the chip has room for, against their solo runs."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,jobs", [(576, 11), (640, 10)])
def test_batched_wide_jobs_equal_their_solo_runs(n, jobs):
    """One full-matrix block per job, ten jobs and more: bit for bit the solo
    results (at these widths the row chunks of the Gram sums are those of the
    solo run)."""
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1507_08751_gb300 import binding as B
    rng = np.random.default_rng(n)
    Y = rng.standard_normal((jobs, n, n))
    for j in range(jobs):
        Y[j] += rng.standard_normal((n, 3)) @ rng.standard_normal((3, n))
    Y = torch.from_numpy(Y.astype(np.float32)).cuda()
    scales, iters = [(1, 1), (n, n)], 4
    X = torch.empty((2, jobs, n, n), device="cuda")
    with B.Context(0) as ctx:
        ctx.msllr_decompose_batch(Y, scales, X, list(range(jobs)), iters=iters)
        for j in range(jobs):
            Xs = torch.empty((2, n, n), device="cuda")
            ctx.msllr_decompose(Y[j].contiguous(), scales, Xs, iters=iters, seed=j)
            torch.cuda.synchronize()
            assert torch.equal(X[:, j], Xs)
            assert Xs.abs().sum() > 0
