"""Back-projection by sums over the grid samples (k_backproject_sum.cu) where it can go wrong:
the first rows it serves (|q| = 0 and the largest), cells of 32 and of 64 rows, a last tile and
cell that are not full, rows whose position is a whole number of samples, one series and a
partial chunk of series.  Whole tables against the oracle, and against the quadrature in the
angle (the direct pipeline) of the same contour."""
import numpy as np
import pytest

import workloads
from tests import cfft_cases as cc

pytestmark = pytest.mark.gpu
TOL = {"fp64": 1e-10, "fp32": 1e-5}


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("n,n_rho,rho_max,q_max", [(1024, 1023, 10.0, 4),     # cells of 64 rows
                                                   (2048, 257, 14.0, 6),      # rows a few samples apart: 32
                                                   (2048, 193, 8.0, 12),      # |q| = 12 starts late
                                                   (1024, 1793, 4.0, 0)])     # many rows per sample
def test_strip_table(precision, n, n_rho, rho_max, q_max):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1404_7357_gb300 import cfft
    wl = workloads.strip_fp64(n=n, n_rho=n_rho, rho_max=rho_max, q_max=q_max)
    wl.precision = precision
    wl.contour.height = min(wl.contour.height, 3.0 / rho_max)
    ctx, got = cc.gpu_table(wl)
    _, ang = cc.gpu_table(wl, options={cfft.OPT_CONTOUR_SERIES: 2})
    ref, _, _ = cc.oracle_table(wl)
    err = cc.rel_err_per_pair(got, ref).max()
    err_ang = cc.rel_err_per_pair(ang, ref).max()
    print(precision, n, n_rho, rho_max, q_max, "sums", err, "angle", err_ang)
    assert err < TOL[precision]


def test_rows_on_whole_samples():
    """rho step of exactly two grid samples: the fractional part is 0 (or just below 1) in every
    row."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    wl = workloads.strip_fp64(n=1024, n_rho=300, rho_max=10.0, q_max=3)
    ctx = cc.gpu_context(wl)
    ds = 2.0 * np.pi / (8.0 * wl.contour.beta_max)
    wl.rho_max = 2.0 * ds * (wl.n_rho - 1)
    ctx, got = cc.gpu_table(wl)
    assert abs(ctx.info()["delta_s"] - ds) < 1e-12 * ds
    ref, _, _ = cc.oracle_table(wl)
    err = cc.rel_err_per_pair(got, ref).max()
    print("whole samples", err)
    assert err < TOL["fp64"]


@pytest.mark.parametrize("m,classes", [(3, 1), (2, 4)])
def test_partial_series_chunks(m, classes):
    """9 and 12 series per harmonic: a chunk of 16 that is not full, rotated classes."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1404_7357_gb300 import cfft
    wl = workloads.patch_m4(n=2048, n_rho=701, rho_max=9.0, q_max=5, rotation_classes=classes)
    wl.element = workloads.patch_rooftops(n_mbf=m)
    _, got = cc.gpu_table(wl)
    _, ang = cc.gpu_table(wl, options={cfft.OPT_CONTOUR_SERIES: 2})
    err = cc.rel_err_per_pair(got, ang.astype(np.complex128)).max()
    print("M", m, "classes", classes, "against the quadrature in the angle", err)
    assert err < 1e-5     # each within 5e-6 of the oracle
