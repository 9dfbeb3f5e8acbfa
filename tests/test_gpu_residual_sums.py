"""The residual sums of the output pass at a size that takes the FP32-pair form
(128 terms per thread and more), against FP64 sums of the returned arrays,
through the C ABI: ordinary values, and values whose squares leave the FP32
range either way.  Bar: a sum of eight terms errs by at most 75 x 2^-48 of it,
the square root by half of that, 1.4e-13, plus the FP64 sums' own rounding."""

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("size", [1.0, 1e-16, 1e18])
def test_residuals_of_a_large_job(size):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1507_08751_gb300 import binding as B
    M, N, L = 4096, 4096, 3
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    assert M * N * L >= 8 * sms * 256 * 128
    g = torch.Generator(device="cuda").manual_seed(5)
    Y = size * torch.randn((M, N), generator=g, device="cuda")
    runs = []
    with B.Context(0) as ctx:
        for iters in (2, 3):
            X = torch.empty((L, M, N), device="cuda")
            Z = torch.empty_like(X)
            st = ctx.msllr_decompose(Y, [(1, 1)] * L, X, iters=iters, seed=3, Z_out=Z,
                                     lambdas=[0.1 * size, 0.2 * size, 0.4 * size])
            runs.append((X, Z, st))
    torch.cuda.synchronize()
    (_, Z0, _), (X, Z, st) = runs
    primal = ((X.double() - Z.double()) ** 2).sum().sqrt().item()
    dual = ((Z.double() - Z0.double()) ** 2).sum().sqrt().item()
    assert primal > 0.0 and dual > 0.0
    assert st["primal_residual"] == pytest.approx(primal, rel=1.5e-13, abs=0.0)
    assert st["dual_residual"] == pytest.approx(dual, rel=1.5e-13, abs=0.0)
