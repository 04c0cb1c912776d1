"""The spectral tables on tall contours (GPU): a contour whose nodes lie many table steps off the
real axis, where a stencil of real nodes extrapolates, keeps the spectra at every node.  Single and
batched tables in both precisions, a patch and the same mesh of radius one, against the direct
pipeline (an explicit series: spectra at every node) within the precision's target; below 1.5 table
steps the tables still serve."""
import dataclasses

import numpy as np
import pytest

import workloads
from tests import cfft_cases as cc

pytestmark = pytest.mark.gpu
TOL = {"fp64": 1e-10, "fp32": 1e-5}


def _workload(element, precision, rho_max, x, n=2048):
    """height * rho_max = x; `element`: "patch", or its mesh of radius 1 ("wide") or 0.66 ("mid": the
    oracle's 128 angles resolve it)."""
    wl = workloads.patch_m4(n=n, n_rho=96, rho_max=rho_max, q_max=3, precision=precision)
    el = workloads.patch_rooftops(n_mbf=2)
    s = {"patch": 1.0, "mid": 1.8, "wide": 2.7}[element]
    wl.element = dataclasses.replace(el, cx=s * el.cx, cy=s * el.cy, half_len=s * el.half_len, width=s * el.width)
    wl.contour.height = x / rho_max
    return wl


def _table(wl, options=None):
    ctx, t = cc.gpu_table(wl, options=options)
    return ctx.info(), t.astype(np.complex128)


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("element,rho_max,x,tables", [("patch", 1.5, 3.0, False), ("patch", 4.0, 3.0, True),
                                                      ("wide", 1.5, 2.25, False), ("wide", 3.0, 3.0, False),
                                                      ("wide", 8.0, 2.0, True)])
def test_single(precision, element, rho_max, x, tables):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1404_7357_gb300 import cfft
    wl = _workload(element, precision, rho_max, x)
    info, got = _table(wl)
    direct, ref = _table(wl, {cfft.OPT_CONTOUR_SERIES: 2})
    err = cc.rel_err_per_pair(got, ref).max()
    print(precision, element, rho_max, x, "against the direct pipeline %.2g" % err)
    assert err < TOL[precision]
    assert (info["work_points"] < direct["work_points"]) == tables


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_single_against_oracle(precision):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    wl = _workload("mid", precision, 1.5, 2.25, n=1536)
    wl.n_rho, wl.q_max = 48, 2
    _, got = _table(wl)
    ref, _, _ = cc.oracle_table(wl)
    err = cc.rel_err_per_pair(got, ref).max()
    print(precision, "radius 0.66 against the oracle %.2g" % err)
    assert err < TOL[precision]


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_batch(precision):
    """Two items, one of them on a low contour: one tall contour keeps the batch off the tables."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1404_7357_gb300 import cfft
    wls = [_workload("wide", precision, 3.0, x) for x in (3.0, 0.1)]
    ctx = cc.gpu_context(wls[0])
    items = [{"eps_r": w.substrate.eps_r, "h": w.substrate.h, "k0": w.substrate.k0, "n": w.contour.n,
              "beta_max": w.contour.beta_max, "beta_p": w.contour.beta_p, "height": w.contour.height,
              "taylor_order": -1} for w in wls]
    prec = cfft.CFFT_FP64 if precision == "fp64" else cfft.CFFT_FP32_MIXED
    out = ctx.tabulate_batch(items, 3, 3.0, 96, prec, graph=True).cpu().numpy()
    for i, w in enumerate(wls):
        _, ref = _table(w, {cfft.OPT_CONTOUR_SERIES: 2})
        err = cc.rel_err_per_pair(out[i][None].astype(np.complex128), ref).max()
        print(precision, "item", i, "batch against the direct pipeline %.2g" % err)
        assert err < TOL[precision]
