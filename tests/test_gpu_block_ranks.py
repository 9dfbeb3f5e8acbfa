"""Block SVT of blocks whose thresholded rank runs through the limits of the
eigen paths (8 pairs up to 64 wide, 16 pairs up to 256 wide), against the FP64
oracle, through the C ABI."""

import numpy as np
import pytest

import oracle as O

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = 1e-4


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1507_08751_gb300 import binding as B
    c = B.Context(0)
    yield c
    c.close()


def _blocks(seed, M, N, m, n, ranks, tau):
    """Dense noise well below tau plus, per block, the given rank of terms with
    singular values between 1.3 and 6 tau."""
    rng = np.random.default_rng(seed)
    A = 0.3 * tau / (np.sqrt(m) + np.sqrt(n)) * rng.standard_normal((M, N))
    i = 0
    for p in range(M // m):
        for q in range(N // n):
            r = min(ranks[i % len(ranks)], m, n)
            i += 1
            if r:
                u, _ = np.linalg.qr(rng.standard_normal((m, r)))
                v, _ = np.linalg.qr(rng.standard_normal((n, r)))
                s = tau * np.exp(rng.uniform(np.log(1.3), np.log(6.0), r))
                A[p * m:(p + 1) * m, q * n:(q + 1) * n] += (u * s) @ v.T
    return A.astype(np.float32)


@pytest.mark.parametrize("m,n", [(17, 17), (33, 40), (48, 64), (64, 64), (120, 60), (65, 65),
                                 (100, 130), (129, 128), (250, 200), (256, 256), (700, 256)])
def test_ranks_around_the_limits(ctx, m, n):
    ranks = (0, 1, 7, 8, 9, 12, 15, 16, 17, 24)
    M, N, tau = 5 * m, 2 * n, 20.0
    A = _blocks(m * 1000 + n, M, N, m, n, ranks, tau)
    Z = torch.full((M, N), float("nan"), dtype=torch.float32, device="cuda")
    rank = torch.empty((10,), dtype=torch.int32, device="cuda")
    ctx.msllr_blocksvt(torch.from_numpy(A).cuda(), Z, m, n, tau, (0, 0), rank_out=rank)
    torch.cuda.synchronize()
    want = O.block_svt(A.astype(np.float64), m, n, tau)
    got = Z.cpu().numpy().astype(np.float64)
    assert np.linalg.norm(got - want) <= TOL * np.linalg.norm(want)
    B = A.astype(np.float64).reshape(5, m, 2, n).transpose(0, 2, 1, 3).reshape(-1, m, n)
    s = np.linalg.svd(B, compute_uv=False)
    near = (np.abs(s - tau) <= 1e-4 * np.maximum(s[:, :1], tau)).any(axis=1)
    assert np.all((rank.cpu().numpy() == (s > tau).sum(axis=1)) | near)
    # block by block, so that a weak block's error is not hidden by a strong one
    for b in range(10):
        p, q = divmod(b, 2)
        sl = np.s_[p * m:(p + 1) * m, q * n:(q + 1) * n]
        assert np.linalg.norm(got[sl] - want[sl]) <= TOL * max(np.linalg.norm(want[sl]), tau)


@pytest.mark.parametrize("m,n,above", [(176, 176, 6), (300, 176, 12), (130, 240, 14), (256, 256, 10),
                                       (120, 100, 9)])
def test_pairs_above_a_crowd_below_tau(ctx, m, n, above):
    """Singular values that crowd just below tau (0.9 .. 0.999 tau) under some
    from 1.002 to 2 tau: slow to converge, must not be taken unconverged.  Bar:
    2e-5 of tau per block entry norm -- the FP32 Gram matrix moves an
    eigenvalue by about n eps lambda_1 = 1e-4 tau^2 at most, a few per cent of
    that in the mean."""
    rng = np.random.default_rng(m + n)
    k, tau = min(m, n), 30.0
    s = np.concatenate([np.linspace(2.0, 1.002, above), np.linspace(0.999, 0.9, k - above)]) * tau
    blocks = []
    for _ in range(4):
        U, _ = np.linalg.qr(rng.standard_normal((m, k)))
        V, _ = np.linalg.qr(rng.standard_normal((n, k)))
        blocks.append((U * s) @ V.T)
    A = np.concatenate(blocks).astype(np.float32)
    Z = torch.empty(A.shape, dtype=torch.float32, device="cuda")
    ctx.msllr_blocksvt(torch.from_numpy(A).cuda(), Z, m, n, tau, (0, 0))
    torch.cuda.synchronize()
    want = O.block_svt(A.astype(np.float64), m, n, tau)
    got = Z.cpu().numpy().astype(np.float64)
    for b in range(4):
        sl = np.s_[b * m:(b + 1) * m]
        assert np.linalg.norm(got[sl] - want[sl]) <= 2e-5 * tau


@pytest.mark.parametrize("m,n", [(33, 33), (40, 40), (40, 100), (48, 64), (60, 60), (64, 64)])
def test_narrow_pairs_above_a_crowd_below_tau(ctx, m, n):
    """Blocks 33 to 64 wide with eight pairs from 1.002 to 1.03 tau over a crowd
    from 0.77 to 0.96 tau, which 32 Lanczos steps do not settle from 40 wide
    on.  Bar per block: settled pairs have residuals of at most 1e-5 lambda_1
    each, so they are exact for a matrix within sqrt(2) sqrt(8) 1e-5 lambda_1
    <= 4.3e-5 tau^2 of G (Frobenius), plus n eps lambda_1 <= 0.9e-5 tau^2 of
    rounding in G; (1 - tau / sqrt(x))_+ has slope 1 / (2 tau^2) at most, so Z
    is within sigma_1 5.2e-5 / 2 = 2.7e-5 tau: 4e-5 tau with the output's own
    rounding."""
    rng = np.random.default_rng(100 * m + n)
    k, tau, nb = min(m, n), 30.0, 16
    s = np.concatenate([np.linspace(1.03, 1.002, 8), np.linspace(0.96, 0.77, k - 8)]) * tau
    blocks = []
    for _ in range(nb):
        U, _ = np.linalg.qr(rng.standard_normal((m, k)))
        V, _ = np.linalg.qr(rng.standard_normal((n, k)))
        blocks.append((U * s) @ V.T)
    A = np.concatenate(blocks).astype(np.float32)
    Z = torch.empty(A.shape, dtype=torch.float32, device="cuda")
    rank = torch.empty((nb,), dtype=torch.int32, device="cuda")
    ctx.msllr_blocksvt(torch.from_numpy(A).cuda(), Z, m, n, tau, (0, 0), rank_out=rank)
    torch.cuda.synchronize()
    want = O.block_svt(A.astype(np.float64), m, n, tau)
    got = Z.cpu().numpy().astype(np.float64)
    assert np.all(rank.cpu().numpy() == 8)
    for b in range(nb):
        sl = np.s_[b * m:(b + 1) * m]
        assert np.linalg.norm(got[sl] - want[sl]) <= 4e-5 * tau


def test_flops_of_a_certified_block_are_its_fp32_steps(ctx):
    """A 256 x 256 noise block of rank 0 above tau: row sums and up to three
    power steps in FP32; the certificate itself runs on the tensor cores."""
    n, tau = 256, 40.0
    A = torch.from_numpy(np.random.default_rng(3).standard_normal((n, n)).astype(np.float32)).cuda()
    X = torch.empty((1, n, n), device="cuda")
    st = ctx.msllr_decompose(A, [(n, n)], X, lambdas=[tau], iters=1, seed=1)
    assert st["blocks_zero"][0] == 1 and st["blocks_householder"][0] == 0
    assert 2 * n * n <= st["flops"][0] <= n + 2 * n * n + 3 * (2 * n * n + 4 * n)


@pytest.mark.parametrize("m,n,kind", [(16, 1024, "full"), (20, 512, "full"), (33, 33, "three"),
                                      (64, 64, "three"), (64, 100, "three"), (100, 100, "three"),
                                      (200, 200, "three")])
def test_what_a_lanczos_breakdown_neglects_is_rounding(ctx, m, n, kind):
    """Blocks whose Krylov space ends after three steps (exact rank three), or is
    used up entirely (14 pairs over two or more equal small values): a coupling
    that the steps neglect must be at rounding level.  Both paths work on the
    same Gram matrix, so the bar is three times the Householder path's own error
    (skip_bound = 0) plus 1e-6 sigma_1 for the rounding of the vectors."""
    from paper_1507_08751_gb300 import binding as B
    k, tau = min(m, n), 10.0
    s = (np.concatenate([np.linspace(6.0, 1.3, 14), np.full(k - 14, 0.2)]) if kind == "full"
         else np.concatenate([[5.0, 3.0, 2.0], np.zeros(k - 3)])) * tau
    for seed in range(12):
        rng = np.random.default_rng(1000 * m + seed)
        U, _ = np.linalg.qr(rng.standard_normal((m, k)))
        V, _ = np.linalg.qr(rng.standard_normal((n, k)))
        want = (U * np.maximum(s - tau, 0.0)) @ V.T
        Y = torch.from_numpy(((U * s) @ V.T).astype(np.float32)).cuda()
        err = []
        for skip in (0, 1):
            p = B.msllr_params_default()
            p.skip_bound = skip
            X = torch.empty((1, m, n), device="cuda")
            Z = torch.empty_like(X)
            ctx.msllr_decompose(Y, [(m, n)], X, lambdas=[tau], iters=1, seed=1, Z_out=Z, params=p)
            err.append(np.linalg.norm(Z[0].double().cpu().numpy() - want))
        assert err[1] <= 3.0 * err[0] + 1e-6 * s[0]
