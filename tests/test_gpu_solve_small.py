"""Reduced systems of one block row and just beyond (GPU): a first block is substituted without its
inverse, one block row runs without a cooperative launch, and the error word comes with the sums.
Orders around the edges (1, a warp, a block, a block and one), both types and refinement.

Tolerances are on the backward error |b - A x|_inf / (|A|_inf |x|_inf + |b|_inf): a few n roundings
of LU with partial pivoting on well-conditioned systems, 4 n 2^-24 (complex64) and 4 n 2^-53
(complex128, and refined, where one rounding of the result is what remains)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch_cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return torch


@pytest.mark.parametrize("dtype,refine", [("complex64", False), ("complex128", False), ("complex128", True)])
def test_backward_error(torch_cuda, dtype, refine):
    torch = torch_cuda
    from paper_1404_7357_gb300 import cfft
    ctx = cfft.Context(0)
    u = 2.0 ** (-24 if dtype == "complex64" else -53)
    for n in (1, 2, 3, 31, 32, 33, 63, 64, 65, 97, 128, 129, 200):
        rng = np.random.default_rng(n)
        a = (rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n))).astype(dtype)
        b = (rng.standard_normal(n) + 1j * rng.standard_normal(n)).astype(dtype)
        za = torch.tensor(a, device="cuda:0")
        x = ctx.solve_reduced(za, torch.tensor(b, device="cuda:0"), refine=refine).cpu().numpy()
        ax, xx = a.astype(np.clongdouble), x.astype(np.clongdouble)
        r = np.abs(b - ax @ xx).max()
        err = float(r / (np.abs(ax).sum(1).max() * np.abs(xx).max() + np.abs(b).max()))
        assert err < 4 * n * u, (n, err / u)
        assert torch.equal(za, torch.tensor(a, device="cuda:0"))


@pytest.mark.parametrize("n", [1, 5, 64, 70])
def test_singular_is_refused_and_the_context_survives(torch_cuda, n):
    torch = torch_cuda
    from paper_1404_7357_gb300 import cfft
    ctx = cfft.Context(0)
    for dtype in (torch.complex64, torch.complex128):
        eye = torch.eye(n, dtype=dtype, device="cuda:0")
        bad = eye.clone()
        bad[n - 1, n - 1] = 0
        v = torch.arange(1, n + 1, device="cuda:0").to(dtype)
        with pytest.raises(cfft.CfftError) as ei:
            ctx.solve_reduced(bad, v)
        assert ei.value.status == 5                       # CFFT_ERR_NUMERIC
        assert torch.equal(ctx.solve_reduced(eye, v), v)
