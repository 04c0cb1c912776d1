"""Line transforms of the Cartesian tabulation at the sizes where they can go wrong: the smallest
grid (several lines per block), powers of two with and without a last radix-2 pass, a line that
fills a block, padded MBF counts; table against the oracle's at fixed orders."""
import numpy as np
import pytest

import workloads
from oracle import cartesian as ocart
from tests import cfft_cases as cc

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,n_grid,order,m", [("fp64", 16, 0, 1), ("fp64", 32, 5, 1), ("fp32", 64, 3, 3),
                                                      ("fp64", 128, 2, 1), ("fp32", 256, 2, 1), ("fp64", 512, 1, 1)])
def test_table_against_oracle(precision, n_grid, order, m):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1404_7357_gb300 import cfft
    wl = workloads.strip_fp64(n=n_grid, n_rho=64, rho_max=2.0, q_max=1)
    if m > 1:
        wl.element = workloads.patch_rooftops(n_side=4, pitch=0.1, n_mbf=m)
    c, s = wl.contour, wl.substrate
    c.beta_p, c.height = 0.26 * c.beta_max, 0.2
    ctx = cc.gpu_context(wl)
    rho = 0.5 * n_grid * np.pi / (2.0 * c.beta_max)
    ctx.tabulate_cartesian(n_grid, rho, cfft.CFFT_FP64 if precision == "fp64" else cfft.CFFT_FP32_MIXED,
                           taylor_order=order)
    got = ctx.cartesian_table().cpu().numpy().astype(np.complex128)
    ref, _ = ocart.table(cc.oracle_basis(wl.element), s.eps_r, s.h, s.k0, c.beta_max, c.beta_p, c.height, n_grid,
                         order)
    ref = ref.reshape(got.shape)
    err = np.abs(got - ref).max() / np.abs(ref).max()
    print(precision, "N", n_grid, "order", order, "M", m, "rel err", err)
    # float64: rounding of two transforms; float32: the spectra's rounding, a few 1e-7
    assert err < (1e-12 if precision == "fp64" else 5e-6)


def test_fill_blocks_of_pairs():
    """67 elements of three MBFs: pairs that do not fill their last block, padded rows, entries
    against the three-point interpolation of the library's own table."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1404_7357_gb300 import cfft
    wl = workloads.strip_fp64(n=64, n_rho=64, rho_max=2.0, q_max=1)
    wl.element = workloads.patch_rooftops(n_side=4, pitch=0.1, n_mbf=3)
    c = wl.contour
    c.beta_p, c.height = 0.26 * c.beta_max, 0.2
    ctx = cc.gpu_context(wl)
    ctx.tabulate_cartesian(64, 1.5, cfft.CFFT_FP64, taylor_order=2)
    tab = ctx.cartesian_table().cpu().numpy()
    inf = ctx.cartesian_info()
    a, m = 67, 3
    pos = np.random.default_rng(2).uniform(-0.5, 0.5, (a, 2))
    z = torch.zeros((a * m, a * m + 5), dtype=torch.complex128, device="cuda:0")
    ctx.fill_cartesian(torch.tensor(pos, device="cuda:0"), z)
    # three-point stencils on the lattice x0 + i step of the table (a lattice rebuilt from its
    # own differences would carry x0's rounding, 64 steps' worth, into the coordinates)
    u = ((pos[:, None] - pos[None]).reshape(-1, 2) - inf["x0"]) / inf["step"]
    i0 = np.floor(u + 0.5).astype(int)
    f = u - i0
    w = np.stack([0.5 * f * (f - 1.0), 1.0 - f * f, 0.5 * f * (f + 1.0)], -1)
    ref = sum(w[:, 0, s] * w[:, 1, r] * tab[:, i0[:, 0] - 1 + s, i0[:, 1] - 1 + r]
              for s in range(3) for r in range(3))
    ref = ref.reshape(m, m, a, a).transpose(2, 0, 3, 1).reshape(a * m, a * m)
    got = z.cpu().numpy()
    assert np.abs(got[:, :a * m] - ref).max() < 1e-13 * np.abs(ref).max()
    assert not got[:, a * m:].any()
