"""The gridded transform and the spectral tables (k_grid.cu) where they can go wrong: contour
lengths that are no power of two (a non-integer number of nodes per coarse cell), a contour on
the real axis (no active nodes), the largest height they serve and the series just beyond it,
and element counts that leave partial blocks of series.  Harmonics and grid against the
oracle's definitions; the grid also against the series of FFTs of the same contour."""
import numpy as np
import pytest

import workloads
from tests import cfft_cases as cc

pytestmark = pytest.mark.gpu


def _strip(n, rho_max, x, q_max, precision):
    """Strip workload with height * rho_max = x (x = 0: the real axis)."""
    wl = workloads.strip_fp64(n=n, n_rho=160, rho_max=rho_max, q_max=q_max)
    wl.precision = precision
    wl.contour.height = x / rho_max
    return wl


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("n,rho_max,x,q_max", [(1024, 10.0, 2.7, 4), (1056, 7.0, 3.5, 3), (1056, 7.0, 3.6, 3),
                                               (3360, 5.3, 1.1, 2), (2048, 4.0, 0.0, 1), (4096, 3.0, 0.3, 0)])
def test_harmonics_and_grid(precision, n, rho_max, x, q_max):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1404_7357_gb300 import cfft
    wl = _strip(n, rho_max, x, q_max, precision)
    nodes, hq = cc.oracle_harmonics(wl)
    c = wl.contour
    # float32: harmonics to a few float32 roundings of their maximum; the transform rounds at
    # about log2(M) 2^-24 of the summed magnitudes, which exp(x) weights at the far end
    tol_y = 1e-12 if precision == "fp64" else 4e-6
    tol_g = 1e-11 if precision == "fp64" else 2e-5
    grids = {}
    for name, opts in (("automatic", {cfft.OPT_BP_KERNEL: 1}),
                       ("series", {cfft.OPT_BP_KERNEL: 1, cfft.OPT_CONTOUR_SERIES: 2})):
        ctx, _ = cc.gpu_table(wl, options=opts)
        info = ctx.info()
        y = ctx.debug_buffer("harmonics").cpu().numpy()[0].astype(np.complex128)
        yref = (hq[0] * (nodes["beta_c"] * nodes["weight"])).reshape(y.shape)
        ey = np.abs(y - yref).max() / np.abs(yref).max()
        k = np.arange(-info["grid_half"], info["grid_half"] + 1)
        s = k * info["delta_s"]
        sel = np.abs(s) <= rho_max
        grid = ctx.debug_buffer("grid").cpu().numpy()[0].astype(np.complex128)[..., sel]
        gref = (yref @ np.exp(-1j * np.outer(nodes["beta_c"], s[sel]))) * np.exp(1j * c.beta_max / 2 * s[sel])
        eg = np.abs(grid - gref).max() / np.abs(gref).max()
        print(precision, name, n, rho_max, x, "harmonics %.2g grid %.2g" % (ey, eg), "FFTs", info["work_subffts"])
        assert ey < tol_y and eg < tol_g
        grids[name] = (info["work_subffts"] * info["sub_len"], info)
    # one transform stands for the series' terms (beyond 3.5 the series itself runs)
    if x <= 3.5:
        assert grids["automatic"][0] < grids["series"][0]
    else:
        assert grids["automatic"][1]["work_subffts"] == grids["series"][1]["work_subffts"]


@pytest.mark.parametrize("m", [1, 3])
def test_patch_series_remainders(m):
    """Series counts that leave partial blocks (9 and 81 series per harmonic block of 8),
    rotated classes, a ragged rho grid, against the direct pipeline's table."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1404_7357_gb300 import cfft
    wl = workloads.patch_m4(n=2080, n_rho=301, rho_max=5.0, q_max=4, rotation_classes=4)
    wl.element = workloads.patch_rooftops(n_mbf=m)
    _, got = cc.gpu_table(wl)
    _, ref = cc.gpu_table(wl, options={cfft.OPT_CONTOUR_SERIES: 2})
    for c in range(4):
        err = cc.rel_err_per_pair(got[c][None], ref[c][None].astype(np.complex128)).max()
        print("M", m, "class", c, "against the direct pipeline", err)
        assert err < 1e-5     # both within 5e-6 of the oracle
