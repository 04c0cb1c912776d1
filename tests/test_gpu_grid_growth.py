"""The gridded transform where its coarse grid is finer than the wanted outputs need (GPU): a
shortest grid of 256 points (1024 in a batch) and a small rho_max make the contour rise many cells,
and the Gaussian's complex weights grow beyond what rounding allows; the series of FFTs serves
there.  Strips at height * rho_max = 3 and more, single and batched, both precisions, against the
series (an explicit CONTOUR_SERIES) and the oracle within the precision's target."""
import numpy as np
import pytest

import workloads
from tests import cfft_cases as cc

pytestmark = pytest.mark.gpu
TOL = {"fp64": 1e-10, "fp32": 1e-5}


def _workload(precision, rho_max, x):
    wl = workloads.strip_fp64(n=2048, n_rho=96, rho_max=rho_max, q_max=3)
    wl.precision = precision
    wl.contour.height = x / rho_max
    return wl


def _table(wl, options=None):
    ctx, t = cc.gpu_table(wl, options=options)
    return ctx.info(), t.astype(np.complex128)


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("rho_max,x,series", [(0.2, 3.0, True), (0.3, 3.0, None), (0.5, 3.0, None), (1.0, 3.5, False),
                                              (2.0, 3.5, False), (4.0, 3.0, False)])
def test_single(precision, rho_max, x, series):
    """series: whether the series of FFTs must run (None: either)."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1404_7357_gb300 import cfft
    wl = _workload(precision, rho_max, x)
    info, got = _table(wl)
    direct, ref = _table(wl, {cfft.OPT_CONTOUR_SERIES: 2})
    oracle, _, _ = cc.oracle_table(wl, rho_index=np.arange(0, wl.n_rho, 5))
    err = cc.rel_err_per_pair(got, ref).max()
    err_o = cc.rel_err_per_pair(got[..., ::5], oracle).max()
    print(precision, rho_max, x, "against the series %.2g the oracle %.2g" % (err, err_o))
    assert err < TOL[precision] and err_o < TOL[precision]
    if series is not None:
        same = info["work_subffts"] * info["sub_len"] == direct["work_subffts"] * direct["sub_len"]
        assert same == series


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("rho_max", [0.3, 0.5, 1.0, 1.5, 2.0])
def test_batch(precision, rho_max):
    """Two items, one of them on a low contour."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1404_7357_gb300 import cfft
    wls = [_workload(precision, rho_max, x) for x in (3.0, 0.1)]
    ctx = cc.gpu_context(wls[0])
    items = [{"eps_r": w.substrate.eps_r, "h": w.substrate.h, "k0": w.substrate.k0, "n": w.contour.n,
              "beta_max": w.contour.beta_max, "beta_p": w.contour.beta_p, "height": w.contour.height,
              "taylor_order": -1} for w in wls]
    prec = cfft.CFFT_FP64 if precision == "fp64" else cfft.CFFT_FP32_MIXED
    out = ctx.tabulate_batch(items, 3, rho_max, 96, prec, graph=True).cpu().numpy()
    for i, w in enumerate(wls):
        _, ref = _table(w, {cfft.OPT_CONTOUR_SERIES: 2})
        err = cc.rel_err_per_pair(out[i][None].astype(np.complex128), ref).max()
        print(precision, rho_max, "item", i, "batch against the series %.2g" % err)
        assert err < TOL[precision]
