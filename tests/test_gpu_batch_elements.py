"""A sweep replayed from its CUDA graph after the element changed (GPU): two elements with the
same basis and MBF counts, the same radius and contours, but three and two rooftop shapes, swept
in turn into the same tables.  Everything a captured launch holds by value must follow the
element; each sweep against single tabulations of the element it was run with."""
import dataclasses

import numpy as np
import pytest

import workloads
from tests import cfft_cases as cc

pytestmark = pytest.mark.gpu
TOL = {"fp32": 1e-5, "fp64": 1e-10}


def _elements(n_mbf):
    """A patch of two shapes, and the same with its inner rooftops narrower (a third and fourth)."""
    two = workloads.patch_rooftops(n_mbf=n_mbf)
    inner = np.hypot(two.cx, two.cy) < 0.12
    more = dataclasses.replace(two, width=np.where(inner, 0.4, 1.0) * two.width)
    return more, two


def _items(n_items):
    out = []
    for i in range(n_items):
        sub = workloads.Substrate(2.2 + i, 0.03 + 0.01 * i)
        c = workloads.default_contour(sub, 2048)
        out.append({"eps_r": sub.eps_r, "h": sub.h, "k0": sub.k0, "n": c.n, "beta_max": c.beta_max,
                    "beta_p": c.beta_p, "height": min(c.height, 0.7), "taylor_order": -1})
    return out


@pytest.mark.parametrize("precision,m,simt", [("fp32", 4, 0), ("fp32", 2, 1), ("fp64", 4, 0), ("fp64", 1, 0)])
def test_graph_follows_the_element(precision, m, simt):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1404_7357_gb300 import cfft
    prec = cfft.CFFT_FP64 if precision == "fp64" else cfft.CFFT_FP32_MIXED
    items, q_max, rho_max, n_rho = _items(2), 3, 4.0, 192
    ctx = cfft.Context(0)
    ctx.set_option(cfft.OPT_SPECTRA_SIMT, simt)
    out = None
    elements = _elements(m)
    for turn, el in enumerate((elements[0], elements[1], elements[0])):
        ctx.set_mbf_spectra(np.stack([el.cx, el.cy], 1), el.direction, el.half_len, el.width, el.q)
        out = ctx.tabulate_batch(items, q_max, rho_max, n_rho, prec, out=out, graph=True)
        got = out.cpu().numpy().astype(np.complex128)
        for i, it in enumerate(items):
            wl = workloads.TableWorkload("element", workloads.Substrate(it["eps_r"], it["h"], it["k0"]), el,
                                         workloads.ContourSpec(it["n"], it["beta_max"], it["beta_p"], it["height"]),
                                         q_max, rho_max, n_rho, precision)
            _, ref = cc.gpu_table(wl, options={cfft.OPT_SPECTRA_SIMT: simt})
            err = cc.rel_err_per_pair(got[i][None], ref.astype(np.complex128)).max()
            print(precision, "M", m, "turn", turn, "item", i, "rel err %.2g" % err)
            assert err < TOL[precision]
