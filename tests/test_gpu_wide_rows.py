"""High harmonics on rho grids whose rows lie many transform samples apart (GPU): the far part of
the back-projection's sample sums is interpolated over cells of rows, and the weights of harmonic q
turn faster over a wide cell the larger q is.  A strip eight wavelengths long on a slab whose
surface waves reach far (its harmonics up to |q| = 60 do not fade along the grid), per harmonic
against the FP64 direct pipeline (the quadrature in the angle).

A row of harmonic q is at most max|g_q| / (2 pi), g_q the transform on the grid, and the sums'
own error is relative to that: float32 1e-7 (end weights), 2e-7 (far interpolation) and roundings,
5e-7 together; FP64 1e-13, 1e-14 and roundings, 1e-12 together; beside what the float32 direct
pipeline is off itself (its spectra and transform).  Harmonics below 1% of the largest are left
out (the strip's odd ones vanish)."""
import numpy as np
import pytest

import workloads
from tests import cfft_cases as cc

pytestmark = pytest.mark.gpu
TOL = {"fp64": 1e-12, "fp32": 5e-7}


@pytest.mark.parametrize("precision,q_max,step,rho_max", [
    ("fp32", 64, 20, 100.0), ("fp32", 64, 5, 100.0), ("fp32", 56, 2.3, 70.0), ("fp32", 48, 1.0, 60.0),
    ("fp32", 32, 20, 60.0), ("fp32", 16, 20, 60.0), ("fp32", 17, 2.5, 40.0),
    ("fp64", 64, 20, 100.0), ("fp64", 56, 9, 70.0), ("fp64", 24, 5, 40.0)])
def test_harmonics(precision, q_max, step, rho_max):
    """step: the rho step in samples of the transform grid."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1404_7357_gb300 import cfft
    wl = workloads.strip_fp64(n=8192, q_max=q_max, rho_max=rho_max)
    wl.element = workloads.strip_element(length=8.0, width=0.3)
    wl.substrate = workloads.Substrate(10.0, 0.1)
    wl.contour = workloads.default_contour(wl.substrate, 8192)
    wl.contour.height = min(wl.contour.height, 1.0 / rho_max)
    ds = 2.0 * np.pi / ((4 if precision == "fp32" else 8) * wl.contour.beta_max)
    wl.n_rho = int(rho_max / (step * ds)) + 1
    direct, ref = cc.gpu_table(wl, options={cfft.OPT_CONTOUR_SERIES: 2})
    g = np.abs(direct.debug_buffer("grid").cpu().numpy()[0, 0]).max(-1) / (2.0 * np.pi)
    wl.precision = precision
    ctx, got = cc.gpu_table(wl)
    _, own = cc.gpu_table(wl, options={cfft.OPT_CONTOUR_SERIES: 2})
    assert abs(ctx.info()["delta_s"] - ds) < 1e-9 * ds
    err = np.abs(got[0, 0].astype(np.complex128) - ref[0, 0]).max(-1)
    err_own = np.abs(own[0, 0].astype(np.complex128) - ref[0, 0]).max(-1)
    q = np.arange(-q_max, q_max + 1)
    seen = g > 0.01 * g.max()
    assert q[seen].max() >= min(q_max, 48) - 1
    over = (err - err_own)[seen] / g[seen]
    print(precision, "q_max", q_max, "step", step, "rows", wl.n_rho, "worst %.2g at q %d"
          % (over.max(), q[seen][over.argmax()]))
    assert over.max() < TOL[precision]


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_batch_takes_the_same_rows(precision):
    """The batched form of a wide grid: the same harmonics by sums and by quadrature."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1404_7357_gb300 import cfft
    wl = workloads.strip_fp64(n=4096, n_rho=150, rho_max=50.0, q_max=24)
    wl.precision = precision
    wl.element = workloads.strip_element(length=4.0, width=0.3)
    wl.contour.height = min(wl.contour.height, 1.0 / wl.rho_max)
    ctx, ref = cc.gpu_table(wl)
    c = wl.contour
    out = ctx.tabulate_batch([{"eps_r": wl.substrate.eps_r, "h": wl.substrate.h, "k0": wl.substrate.k0, "n": c.n,
                               "beta_max": c.beta_max, "beta_p": c.beta_p, "height": c.height, "taylor_order": -1}],
                             wl.q_max, wl.rho_max, wl.n_rho,
                             cfft.CFFT_FP64 if precision == "fp64" else cfft.CFFT_FP32_MIXED)
    err = cc.rel_err_per_pair(out.cpu().numpy()[0][None], ref.astype(np.complex128)).max()
    print(precision, "batch against single %.2g" % err)
    assert err < (1e-12 if precision == "fp64" else 2e-6)
