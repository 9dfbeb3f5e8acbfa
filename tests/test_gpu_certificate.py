"""The certificate of blocks wider than 256 (no singular value above tau
outside the kept pairs), through the C ABI: orders at the edges of its 64- and
128-wide tiles, a flat spectrum just below tau, and a block that must not be
certified."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1507_08751_gb300 import binding as B
    c = B.Context(0)
    yield c
    c.close()


def _with_spectrum(seed, M, N, s):
    rng = np.random.default_rng(seed)
    k = len(s)
    U, _ = np.linalg.qr(rng.standard_normal((M, k)))
    V, _ = np.linalg.qr(rng.standard_normal((N, k)))
    return ((U * s) @ V.T).astype(np.float32)


def _one_svt(ctx, A, tau):
    X = torch.empty((1,) + A.shape, dtype=torch.float32, device="cuda")
    Z = torch.empty_like(X)
    st = ctx.msllr_decompose(torch.from_numpy(A).cuda(), [A.shape], X, lambdas=[tau], rho=1.0,
                             iters=1, seed=1, Z_out=Z)
    torch.cuda.synchronize()
    return Z[0].cpu().numpy().astype(np.float64), st


@pytest.mark.parametrize("M,N", [(257, 257), (320, 400), (384, 321), (700, 511), (513, 640),
                                 (1100, 1025)])
def test_flat_spectrum_below_tau_is_certified(ctx, M, N):
    """Every singular value outside three strong ones is 0.96 tau: the power
    sum bound exceeds the largest eigenvalue by n^(1/512) <= 1.4 % and the
    rounding terms by less than 2 %, so 0.9216 tau^2 is certified."""
    n, tau = min(M, N), 50.0
    s = np.concatenate([[400.0, 200.0, 100.0], np.full(n - 3, 0.96 * tau)])
    A = _with_spectrum(M + N, M, N, s)
    got, st = _one_svt(ctx, A, tau)
    assert st["blocks_uncertified"][0] == 0
    assert st["blocks_lanczos"][0] == 1
    U, sv, Vt = np.linalg.svd(A.astype(np.float64), full_matrices=False)
    want = (U * np.maximum(sv - tau, 0)) @ Vt
    assert np.linalg.norm(got - want) <= 1e-4 * np.linalg.norm(want)


@pytest.mark.parametrize("M,N", [(300, 300), (520, 1030)])
def test_more_pairs_than_kept_is_not_certified(ctx, M, N):
    """20 singular values above tau: at most 16 pairs are kept, so the
    certificate has to fail."""
    s = np.concatenate([np.linspace(200.0, 100.0, 20), np.full(50, 1.0)])
    _, st = _one_svt(ctx, _with_spectrum(M, M, N, s), 50.0)
    assert st["blocks_uncertified"][0] == 1
