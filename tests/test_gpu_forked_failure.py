"""A call that stops while its second stream is forked (GPU; the failure is injected on the host, no
launch of it is bad): the status is CFFT_ERR_CUDA, the second stream is joined again (a capture
ends with it, too), and the next calls on the same context give what a fresh context gives: to the
bit, FP64 tables to the roundings of their low rows (atomic sums in any order, 1e-13 of the table)."""
import numpy as np
import pytest

import workloads
from tests import cfft_cases as cc

pytestmark = pytest.mark.gpu


@pytest.fixture()
def lib():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1404_7357_gb300 import cfft
    yield torch, cfft
    cfft.test_fail_forked_launch(-1)


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_tabulation(lib, precision):
    torch, cfft = lib
    wl = cc.small_patch(precision, n=1024, n_rho=512, rho_max=6.0, q_max=3)
    prec = cfft.CFFT_FP64 if precision == "fp64" else cfft.CFFT_FP32_MIXED
    _, ref = cc.gpu_table(wl)
    ctx = cc.gpu_context(wl)
    for _ in range(3):
        cfft.test_fail_forked_launch(0)
        with pytest.raises(cfft.CfftError) as ei:
            ctx.tabulate_reactions(wl.q_max, wl.rho_max, wl.n_rho, prec, 1)
        assert ei.value.status == 4                      # CFFT_ERR_CUDA
        ctx.tabulate_reactions(wl.q_max, wl.rho_max, wl.n_rho, prec, 1)
        got = ctx.copy_table(host=True).numpy()
        assert np.abs(got - ref).max() <= (1e-13 if precision == "fp64" else 0.0) * np.abs(ref).max()


@pytest.mark.parametrize("graph", [False, True])
def test_batch(lib, graph):
    torch, cfft = lib
    el = workloads.patch_rooftops()
    items = []
    for eps in (2.2, 4.4):
        sub = workloads.Substrate(eps, 0.03)
        c = workloads.default_contour(sub, 1024)
        items.append({"eps_r": eps, "h": 0.03, "k0": sub.k0, "n": 1024, "beta_max": c.beta_max, "beta_p": c.beta_p,
                      "height": 0.4, "taylor_order": -1})

    def run(ctx):
        return ctx.tabulate_batch(items, 3, 6.0, 512, cfft.CFFT_FP32_MIXED, graph=graph).cpu().numpy()

    def context():
        ctx = cfft.Context(0)
        ctx.set_mbf_spectra(np.stack([el.cx, el.cy], 1), el.direction, el.half_len, el.width, el.q)
        return ctx
    ref = run(context())
    ctx = context()
    for _ in range(2):
        cfft.test_fail_forked_launch(0)
        with pytest.raises(cfft.CfftError) as ei:
            run(ctx)
        assert ei.value.status == 4
        cfft.test_fail_forked_launch(-1)
        assert np.array_equal(run(ctx), ref)


def test_factorization(lib):
    torch, cfft = lib
    n = 3400                     # five panels look ahead
    gen = torch.Generator(device="cuda:0").manual_seed(3)
    z = torch.randn((n, n), dtype=torch.complex64, device="cuda:0", generator=gen)
    z += 60.0 * torch.eye(n, device="cuda:0")
    v = torch.randn(n, dtype=torch.complex64, device="cuda:0", generator=gen)
    ctx = cfft.Context(0)
    ref = ctx.solve_reduced(z, v)
    for after in (0, 2):
        cfft.test_fail_forked_launch(after)
        with pytest.raises(cfft.CfftError) as ei:
            ctx.solve_reduced(z, v)
        assert ei.value.status == 4
        assert torch.equal(ctx.solve_reduced(z, v), ref)
