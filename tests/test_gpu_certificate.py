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


def _cold_svts(ctx, blocks, tau):
    """One iteration on a stack of blocks, moved so that the shifted grid meets
    them: not the full matrix, so every block starts from the cold basis."""
    from paper_1507_08751_gb300 import binding as B
    A = np.concatenate(blocks)
    sr, sc = (int(v) for v in B.msllr_shift_table(1, 1, *A.shape)[0])
    X = torch.empty((1,) + A.shape, dtype=torch.float32, device="cuda")
    Z = torch.empty_like(X)
    Y = np.ascontiguousarray(np.roll(A, (sr, sc), (0, 1)), dtype=np.float32)
    st = ctx.msllr_decompose(torch.from_numpy(Y).cuda(), [blocks[0].shape], X, lambdas=[tau], rho=1.0,
                             iters=1, seed=1, Z_out=Z)
    torch.cuda.synchronize()
    got = np.roll(Z[0].cpu().numpy().astype(np.float64), (-sr, -sc), (0, 1))
    return np.split(got, len(blocks)), st


@pytest.mark.parametrize("M,N,above", [(257, 300, 8), (300, 300, 8), (512, 600, 12), (1030, 1030, 6),
                                       (2100, 2100, 6)])
def test_slow_pairs_above_a_crowd_below_tau(ctx, M, N, above):
    """Pairs from 1.002 to 1.3 tau over a crowd from 0.88 to 0.93 tau: the basis
    gains a factor of 0.87 a step for the weakest, some 50 steps in all.  A block whose pairs
    have not converged must not count as certified.  Bar: converged pairs have
    residuals of at most 3e-4 tau^2 each, so they are exact for a matrix within
    sqrt(2 k) 3e-4 tau^2 of G; (1 - tau / sqrt(x))_+ has slope 1 / (2 tau^2) at
    most, so Z is within 1.3 sqrt(2 k) 1.5e-4 tau, plus the same factor times
    G's rounding, n eps lambda_1 <= 2e-7 n tau^2."""
    n, tau = min(M, N), 50.0
    s = np.concatenate([np.linspace(1.3, 1.002, above), np.linspace(0.93, 0.8835, n - above)]) * tau
    rng = np.random.default_rng(M + N)
    blocks, want = [], []
    for _ in range(2):
        U, _ = np.linalg.qr(rng.standard_normal((M, n)))
        V, _ = np.linalg.qr(rng.standard_normal((N, n)))
        blocks.append((U * s) @ V.T)
        want.append((U * np.maximum(s - tau, 0.0)) @ V.T)
    got, st = _cold_svts(ctx, blocks, tau)
    assert st["blocks_uncertified"][0] == 0
    assert st["blocks_lanczos"][0] == 2
    bar = 1.3 * (np.sqrt(2 * above) * 1.5e-4 + 1e-7 * n) * tau
    for g, w in zip(got, want):
        assert np.linalg.norm(g - w) <= bar


def test_pairs_slower_than_every_round_count_as_uncertified(ctx):
    """Pairs at 1.002 tau over forty at 0.995 tau: 0.986 a step, not settled in
    any number of steps that is run."""
    n, tau = 320, 50.0
    s = np.concatenate([np.full(4, 1.002), np.full(40, 0.995), np.full(n - 44, 0.3)]) * tau
    rng = np.random.default_rng(n)
    blocks = []
    for _ in range(2):
        U, _ = np.linalg.qr(rng.standard_normal((n, n)))
        V, _ = np.linalg.qr(rng.standard_normal((n, n)))
        blocks.append((U * s) @ V.T)
    _, st = _cold_svts(ctx, blocks, tau)
    assert st["blocks_uncertified"][0] == 2


def test_slow_pairs_of_many_blocks(ctx):
    """The further rounds in the form for launches that fill the chip: ten
    blocks and more, as test_slow_pairs_above_a_crowd_below_tau."""
    n, above, tau = 260, 6, 50.0
    s = np.concatenate([np.linspace(1.3, 1.002, above), np.linspace(0.93, 0.8835, n - above)]) * tau
    rng = np.random.default_rng(n)
    blocks, want = [], []
    for _ in range(12):
        U, _ = np.linalg.qr(rng.standard_normal((n, n)))
        V, _ = np.linalg.qr(rng.standard_normal((n, n)))
        blocks.append((U * s) @ V.T)
        want.append((U * np.maximum(s - tau, 0.0)) @ V.T)
    got, st = _cold_svts(ctx, blocks, tau)
    assert st["blocks_uncertified"][0] == 0
    bar = 1.3 * (np.sqrt(2 * above) * 1.5e-4 + 1e-7 * n) * tau
    for g, w in zip(got, want):
        assert np.linalg.norm(g - w) <= bar


@pytest.mark.parametrize("M,N", [(257, 257), (320, 300), (512, 512), (1024, 1024)])
def test_many_pairs_are_as_accurate_as_few(ctx, M, N):
    """Fourteen pairs from 1.3 to 6 tau: the rotations of the 32 x 32 Ritz problem
    must not leave the vectors off unit length.  Bar per block: 8 eps ||Z||_F --
    two eps for the length of u on either side of the product, as much again
    for the rounding of G (an eigenvalue's counts half in sigma) and of the
    products."""
    n, tau = min(M, N), 10.0
    s = np.concatenate([np.linspace(6.0, 1.3, 14), np.full(n - 14, 0.2)]) * tau
    rng = np.random.default_rng(M + N)
    blocks, want = [], []
    for _ in range(4):
        U, _ = np.linalg.qr(rng.standard_normal((M, n)))
        V, _ = np.linalg.qr(rng.standard_normal((N, n)))
        blocks.append((U * s) @ V.T)
        want.append((U * np.maximum(s - tau, 0.0)) @ V.T)
    got, st = _cold_svts(ctx, blocks, tau)
    assert st["blocks_uncertified"][0] == 0
    for g, w in zip(got, want):
        assert np.linalg.norm(g - w) <= 8 * 2.0 ** -23 * np.linalg.norm(w)
