"""The solve at the edges of its panel forms and substitution (GPU).

- Panels of more than 2048 rows run as two halves, whole or half on one thread-block cluster
  where its shared memory holds the rows (halves: 12,880 rows in complex64, 6,032 in
  complex128), else over the grid: the same pivots and operations, so the solution equals that
  of the grid form (option SOLVE_GRID_PANEL) to the bit.
- The substitutions at one block of 64, its neighbours, ragged last blocks and more blocks than
  the device has SMs, against the residual bound of a stable solve: |b - A x| is at most
  c n eps |A| |x| with a small c; with entries of order 1 and c = 8 in the 2-norm bounded by
  Frobenius' norm.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch_cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    return torch


def _system(torch, n, dtype, seed):
    g = torch.Generator(device="cuda:0").manual_seed(seed)
    real = torch.float32 if dtype == torch.complex64 else torch.float64
    a = torch.complex(*(torch.randn((n, n), generator=g, device="cuda:0", dtype=real) for _ in range(2)))
    b = torch.complex(*(torch.randn((n,), generator=g, device="cuda:0", dtype=real) for _ in range(2)))
    a.diagonal().zero_()      # every column exchanges rows
    return a, b


def _residual_ok(torch, a, b, x, eps):
    n = a.shape[0]
    r = b.to(torch.complex128)
    for i in range(0, n, 1024):
        r[i:i + 1024] -= a[i:i + 1024].to(torch.complex128) @ x.to(torch.complex128)
    scale = float(torch.linalg.vector_norm(a)) * float(torch.linalg.vector_norm(x))
    return float(torch.linalg.vector_norm(r)) <= 8.0 * eps * np.sqrt(n) * scale


@pytest.mark.parametrize("n,dtype", [(2049, "complex64"), (2112, "complex128"), (6100, "complex128"),
                                     (12950, "complex64")])
def test_half_panels_cluster_against_grid(torch_cuda, n, dtype):
    torch = torch_cuda
    from paper_1404_7357_gb300 import cfft
    a, b = _system(torch, n, getattr(torch, dtype), n)
    xs = []
    for grid in (0, 1):
        ctx = cfft.Context(0)
        ctx.set_option(cfft.OPT_SOLVE_GRID_PANEL, grid)
        xs.append(ctx.solve_reduced(a, b).clone())
        del ctx
    assert torch.equal(xs[0], xs[1])
    assert _residual_ok(torch, a, b, xs[0], 6e-8 if dtype == "complex64" else 1.2e-16)


@pytest.mark.parametrize("dtype", ["complex64", "complex128"])
@pytest.mark.parametrize("n", [1, 63, 64, 65, 200, 9800])
def test_substitution_blocks(torch_cuda, n, dtype):
    torch = torch_cuda
    from paper_1404_7357_gb300 import cfft
    if n == 9800 and dtype == "complex128":
        pytest.skip("the block rule does not depend on the type")
    a, b = _system(torch, n, getattr(torch, dtype), 3 + n)
    if n == 1:
        a.fill_(2.0 - 1.0j)
    ctx = cfft.Context(0)
    x = ctx.solve_reduced(a, b)
    assert _residual_ok(torch, a, b, x, 6e-8 if dtype == "complex64" else 1.2e-16)
