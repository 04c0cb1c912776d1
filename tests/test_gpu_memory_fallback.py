"""A tabulation or a batch without memory for the gridded transform, the spectral tables or the sample
sums runs the direct pipeline, which needs none of their buffers (GPU; the failure is injected on
the host): for every allocation of a fresh context's first call, the call reports CFFT_ERR_OOM or
returns the table within the precision's target, and at least the buffers that the direct pipeline
does without fall back."""
import numpy as np
import pytest

import workloads
from tests import cfft_cases as cc

pytestmark = pytest.mark.gpu
TOL = {"fp64": 1e-10, "fp32": 1e-5}


@pytest.fixture()
def lib():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1404_7357_gb300 import cfft
    yield cfft
    cfft.test_fail_allocation(-1)


def _outcomes(cfft, count, context, run, work, ref, tol):
    """Statuses of the first call with each of the first `count` allocations failing: "oom", or the
    work the call reports."""
    out = []
    for after in range(count):
        ctx = context()
        cfft.test_fail_allocation(after)
        try:
            got = run(ctx)
        except cfft.CfftError as e:
            assert e.status == 3
            out.append("oom")
            got = run(ctx)                      # the context is usable
        else:
            out.append(work(ctx))
        finally:
            cfft.test_fail_allocation(-1)
        assert np.abs(got - ref).max() < tol * np.abs(ref).max(), after
    return out


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_tabulation(lib, precision):
    cfft = lib
    wl = cc.small_patch(precision, n=1024, n_rho=512, rho_max=6.0, q_max=3)
    prec = cfft.CFFT_FP64 if precision == "fp64" else cfft.CFFT_FP32_MIXED

    def run(ctx):
        ctx.tabulate_reactions(wl.q_max, wl.rho_max, wl.n_rho, prec, 1)
        return ctx.copy_table(host=True).numpy()
    direct, ref = cc.gpu_table(wl, options={cfft.OPT_CONTOUR_SERIES: 2})
    auto, _ = cc.gpu_table(wl)
    w_direct, w_auto = direct.info()["work_points"], auto.info()["work_points"]
    assert w_auto < w_direct
    out = _outcomes(cfft, 24, lambda: cc.gpu_context(wl), run, lambda c: c.info()["work_points"], ref, TOL[precision])
    print(precision, out)
    assert out.count(w_direct) == 5             # weights, coarse samples, nodes, tables, sums
    assert set(out) <= {"oom", w_direct, w_auto} and out[0] == "oom"


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_batch(lib, precision):
    cfft = lib
    el = workloads.patch_rooftops()
    prec = cfft.CFFT_FP64 if precision == "fp64" else cfft.CFFT_FP32_MIXED
    items = []
    for eps in (2.2, 4.4):
        sub = workloads.Substrate(eps, 0.03)
        c = workloads.default_contour(sub, 1024)
        items.append({"eps_r": eps, "h": 0.03, "k0": sub.k0, "n": 1024, "beta_max": c.beta_max, "beta_p": c.beta_p,
                      "height": 0.4, "taylor_order": -1})

    def context(series=0):
        ctx = cfft.Context(0)
        ctx.set_mbf_spectra(np.stack([el.cx, el.cy], 1), el.direction, el.half_len, el.width, el.q)
        ctx.set_option(cfft.OPT_CONTOUR_SERIES, series)
        return ctx

    def run(ctx):
        return ctx.tabulate_batch(items, 3, 6.0, 512, prec, graph=True).cpu().numpy()

    def work(ctx):
        return ctx.batch_info()["work_subffts"]
    direct, auto = context(2), context()
    ref = run(direct)
    run(auto)
    assert work(auto) < work(direct)
    out = _outcomes(cfft, 40, context, run, work, ref, TOL[precision])
    print(precision, out)
    assert out.count("oom") + sum(w in (work(direct), work(auto)) for w in out) == len(out)
    assert sum(w == work(direct) for w in out) == 4     # coarse samples, weights, sums, tables
