"""The FP64 bucketed fill's windows shared by one to eight CTAs (GPU), where the shares can go wrong: one
and two CTAs of shared memory per SM, enough windows that none is shared, empty windows, windows
of fewer pairs than threads (items are MBF rows) and of many, one and four classes, M = 1, 2, 4;
against the per-row form, whose order of sums differs (1e-12 of the matrix, as the forms' other
comparisons)."""
import numpy as np
import pytest

import workloads
from tests import cfft_cases as cc

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,classes,q_max,n_rho,elements", [
    (4, 1, 16, 2048, 260),    # one CTA per SM, more windows than SMs
    (4, 1, 16, 96, 260),      # one CTA per SM, few windows
    (4, 4, 8, 4096, 70),      # more windows than eight CTAs per SM
    (4, 1, 8, 300, 300),      # dense windows
    (2, 4, 6, 900, 120), (2, 1, 3, 64, 250), (1, 4, 4, 2500, 150), (1, 1, 0, 200, 400)])
def test_shares_against_the_per_row_form(m, classes, q_max, n_rho, elements):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1404_7357_gb300 import cfft
    rho_max = 9.0
    wl = cc.small_patch("fp64", n=1024, n_rho=n_rho, rho_max=rho_max, q_max=q_max, rotation_classes=classes)
    wl.element = workloads.patch_rooftops(n_mbf=m)
    ctx, _ = cc.gpu_table(wl, options={cfft.OPT_FILL_REFINE: 1})
    rng = np.random.default_rng(elements)
    # uneven over the distances: a dense patch and a sparse ring
    r = np.where(np.arange(elements) % 3 == 0, 4.4, 0.7) * np.sqrt(rng.uniform(0.1, 1.0, elements))
    t = rng.uniform(0, 2 * np.pi, elements)
    pos = torch.tensor(np.stack([r * np.cos(t), r * np.sin(t)], -1), device="cuda:0")
    rot = torch.tensor(workloads.rotations(elements, seed=7), device="cuda:0") if classes == 4 else None
    out = {}
    for block in (0, -1):
        ctx.set_option(cfft.OPT_FILL_BLOCK, block)
        z = torch.full((elements * m, elements * m), 7.0, dtype=torch.complex128, device="cuda:0")
        ctx.fill_reduced_matrix(pos, rot, z)
        out[block] = (z, ctx.info()["fill_form"])
    assert (out[0][1], out[-1][1]) == (2, 1)
    err = ((out[0][0] - out[-1][0]).abs().max() / out[-1][0].abs().max()).item()
    print(m, classes, q_max, n_rho, elements, "rel err %.2g" % err)
    assert err < 1e-12
