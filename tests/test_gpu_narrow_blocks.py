"""Block SVT of the narrowest blocks (several per warp up to 8 x 16), through
the C ABI against the FP64 oracle: every lane and row count at its edges,
block counts that leave the last warp partly empty, shifts that wrap, blocks
that are zero, constant or exactly rank deficient.  Bar per block: 1e-5 of
max(sigma_1, tau), a few times the rotation tolerance (2e-6) that the columns
are orthogonalised to."""

import numpy as np
import pytest

import oracle as O

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


@pytest.mark.parametrize("m,n", [(1, 2), (2, 1), (2, 2), (3, 3), (4, 4), (4, 5), (8, 4), (3, 8),
                                 (4, 9), (5, 5), (8, 8), (7, 13), (16, 8), (8, 16), (1, 16),
                                 (9, 9), (8, 17)])
def test_narrow_blocks_match_oracle(ctx, m, n):
    rng = np.random.default_rng(100 * m + n)
    bm, bn = 7, 5
    M, N = bm * m, bn * n
    A = 0.2 * rng.standard_normal((M, N))
    for p in range(bm):
        for q in range(bn):
            kind = (p * bn + q) % 6
            blk = np.s_[p * m:(p + 1) * m, q * n:(q + 1) * n]
            if kind == 0:
                A[blk] = 0.0
            elif kind == 1:
                A[blk] = 1.5  # rank one, equal columns
            elif kind == 2:
                A[blk] += 3.0 * np.outer(rng.standard_normal(m), rng.standard_normal(n))
            elif kind == 3:
                A[blk] = 40.0 * rng.standard_normal((m, n))  # every pair above tau
            elif kind == 4:
                A[blk] += np.outer(rng.standard_normal(m), rng.standard_normal(n)) * 30.0
    A = A.astype(np.float32)
    tau = 0.8 * (np.sqrt(m) + np.sqrt(n))
    for shift in ((0, 0), (M - 1, 1)):
        Z = torch.full((M, N), float("nan"), dtype=torch.float32, device="cuda")
        rank = torch.full((bm * bn,), -1, dtype=torch.int32, device="cuda")
        ctx.msllr_blocksvt(torch.from_numpy(A).cuda(), Z, m, n, float(tau), shift, rank_out=rank)
        torch.cuda.synchronize()
        A64 = O.shift(A.astype(np.float64), shift)
        want = O.block_svt(A64, m, n, tau)
        got = O.shift(Z.cpu().numpy().astype(np.float64), shift)
        B = A64.reshape(bm, m, bn, n).transpose(0, 2, 1, 3).reshape(-1, m, n)
        s = np.linalg.svd(B, compute_uv=False)
        near = (np.abs(s - tau) <= 1e-4 * np.maximum(s[:, :1], tau)).any(axis=1)
        assert np.all((rank.cpu().numpy() == (s > tau).sum(axis=1)) | near)
        for b in range(bm * bn):
            p, q = divmod(b, bn)
            blk = np.s_[p * m:(p + 1) * m, q * n:(q + 1) * n]
            assert np.linalg.norm(got[blk] - want[blk]) <= 1e-5 * max(s[b, 0], tau)


@pytest.mark.parametrize("n", [4, 8, 16])
def test_narrow_blocks_with_pairs_on_both_sides_of_tau(ctx, n):
    """Singular values 1.04 and 0.946 tau and small ones: rotations that leave
    the columns below tau alone converge slowly here, the result must not
    depend on it.  Bar per block as above, halved: 5e-6."""
    rng = np.random.default_rng(n)
    nb, tau = 2048, 3.0
    s = np.full(n, 0.03)
    s[:4] = (1.043, 0.9458, 0.1926, 0.0669)
    U, _ = np.linalg.qr(rng.standard_normal((nb, n, n)))
    V, _ = np.linalg.qr(rng.standard_normal((nb, n, n)))
    A = ((U * (s * tau)) @ V.transpose(0, 2, 1)).astype(np.float32)
    Z = torch.empty((nb * n, n), dtype=torch.float32, device="cuda")
    ctx.msllr_blocksvt(torch.from_numpy(A.reshape(nb * n, n)).cuda(), Z, n, n, tau, (0, 0))
    torch.cuda.synchronize()
    u, sv, vt = np.linalg.svd(A.astype(np.float64))
    want = (u * np.maximum(sv - tau, 0.0)[:, None, :]) @ vt
    err = np.linalg.norm(Z.cpu().numpy().astype(np.float64).reshape(nb, n, n) - want, axis=(1, 2))
    assert np.all(err <= 5e-6 * sv[:, 0])
