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


def test_blocks_just_above_256_fit_the_budget_they_always_had():
    """102 blocks of 257 x 257 (one row chunk of the Gram sums each) within the
    bytes that two FP32 matrices, the Gram partials and the bases take; first
    and last block against FP64."""
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1507_08751_gb300 import binding as B
    n, nb, tau = 257, 102, 40.0
    M, N = n * nb // 2, 2 * n
    tiles = 15
    need = nb * (4 * tiles * 4096 + 8 * n * n + 8 * tiles + 8 * n * 32 + 12 * n * 16 + 104) + 4096
    g = torch.Generator(device="cuda").manual_seed(7)
    A = torch.randn((M, N), generator=g, device="cuda")
    A += torch.randn((M, 2), generator=g, device="cuda") @ torch.randn((2, N), generator=g, device="cuda")
    Z = torch.empty_like(A)
    with B.Context(0, (need + 255) // 256 * 256 + 256) as ctx:
        ctx.msllr_blocksvt(A, Z, n, n, tau, (0, 0))
    torch.cuda.synchronize()
    for sl in (np.s_[:n, :n], np.s_[M - n:, n:]):
        U, s, Vt = np.linalg.svd(A[sl].double().cpu().numpy(), full_matrices=False)
        want = (U * np.maximum(s - tau, 0.0)) @ Vt
        assert np.linalg.norm(Z[sl].double().cpu().numpy() - want) <= 1e-4 * np.linalg.norm(want)
