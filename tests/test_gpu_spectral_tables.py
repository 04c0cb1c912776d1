"""The spectral tables' kernel (real nodes; D and E from one spectrum) where it can go wrong (GPU),
against the per-node spectra of the direct pipeline: every padded MBF count, one and four rotation
classes, harmonics in every residue class, few and many angles, basis centres on a mesh (tabulated
coordinate factors) and off it (a sine and cosine each).

Tolerances: float64 1e-11 of the table (interpolation 1e-14, sums of 200 terms and the transform
a few hundred roundings each), float32 1e-5, the precision's target for either pipeline.
"""
import dataclasses

import numpy as np
import pytest

import workloads
from tests import cfft_cases as cc

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,m,classes,q_max,n_alpha,mesh", [
    ("fp64", 1, 4, 3, 0, True), ("fp64", 2, 1, 0, 128, False), ("fp64", 3, 4, 5, 256, True),
    ("fp64", 4, 1, 2, 0, False), ("fp64", 8, 1, 4, 0, True), ("fp32", 8, 4, 3, 0, True),
    ("fp32", 4, 1, 6, 256, True), ("fp32", 2, 4, 1, 0, False)])
def test_tables_against_direct(precision, m, classes, q_max, n_alpha, mesh):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1404_7357_gb300 import cfft
    wl = workloads.patch_m4(n=2048, n_rho=161, rho_max=4.0, q_max=q_max, precision=precision, rotation_classes=classes)
    el = workloads.patch_rooftops(n_mbf=m)
    if not mesh:
        rng = np.random.default_rng(m)
        el = dataclasses.replace(el, cx=el.cx + 1e-3 * rng.standard_normal(len(el.cx)),
                                 cy=el.cy + 1e-3 * rng.standard_normal(len(el.cy)))
    wl.element = el
    opts = {cfft.OPT_SPECTRA_SIMT: 1}
    if n_alpha:
        opts[cfft.OPT_N_ALPHA] = n_alpha
    _, got = cc.gpu_table(wl, options=opts)
    _, ref = cc.gpu_table(wl, options={**opts, cfft.OPT_CONTOUR_SERIES: 2})
    for c in range(classes):
        err = cc.rel_err_per_pair(got[c][None], ref[c][None].astype(np.complex128)).max()
        print(precision, m, classes, c, "%.2g" % err)
        assert err < (1e-11 if precision == "fp64" else 1e-5)
