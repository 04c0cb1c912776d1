"""The fill of few pairs straight from the table (GPU) against the sorted fill (option FILL_BLOCK
set): M in {1, 2, 4}, 8, 12 and 16 taps, one and four rotation classes, odd leading dimensions,
one element up to the last count of the rule, the parity rows, and a pair beyond the table.

The two forms take the same stencils and weights and sum taps and harmonics in another order:
at most 16 taps times 17 harmonics, a few units in the last place of the largest term, 2e-6 and
1e-13 of the matrix maximum."""
import dataclasses

import numpy as np
import pytest

import workloads
from tests import cfft_cases as cc

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch_cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return torch


def _fill(torch, ctx, pos, rot, m, dt, block, pad=0):
    from paper_1404_7357_gb300 import cfft
    a = len(pos)
    ctx.set_option(cfft.OPT_FILL_BLOCK, block)
    z = torch.full((a * m, a * m + pad), 7.0, dtype=dt, device="cuda:0")
    rt = None if rot is None else torch.tensor(rot, device="cuda:0")
    ctx.fill_reduced_matrix(torch.tensor(pos, device="cuda:0"), rt, z)
    form = ctx.info()["fill_form"]
    out = z.cpu().numpy()
    assert np.all(out[:, a * m:] == 7.0)
    return out[:, :a * m], form


@pytest.mark.parametrize("precision,m,taps,classes", [("fp32", 4, 8, 4), ("fp32", 2, 8, 1), ("fp32", 1, 12, 4),
                                                      ("fp64", 4, 16, 4), ("fp64", 2, 12, 1), ("fp64", 1, 16, 1)])
def test_direct_against_sorted(torch_cuda, precision, m, taps, classes):
    torch = torch_cuda
    from paper_1404_7357_gb300 import cfft
    wl = cc.small_patch(precision, n=1024, n_rho=1024, rho_max=9.0, q_max=8, rotation_classes=classes)
    el = wl.element
    wl = dataclasses.replace(wl, element=dataclasses.replace(el, q=np.ascontiguousarray(el.q[:, :m])))
    ctx, _ = cc.gpu_table(wl, options={cfft.OPT_FILL_TAPS: taps})
    dt = torch.complex128 if precision == "fp64" else torch.complex64
    last = 45 if precision == "fp64" else 78        # 45^2 <= 2048 < 46^2, 78^2 <= 6144 < 79^2
    for a, pad in ((1, 0), (2, 1), (last, 3), (last + 1, 0)):
        pos = workloads.poisson_disc(a, 4.4, 0.3, seed=31)
        rot = workloads.rotations(a, seed=31) if classes == 4 else None
        got, form = _fill(torch, ctx, pos, rot, m, dt, 0, pad)
        assert (form == 4) == (a <= last)
        ref, sorted_form = _fill(torch, ctx, pos, rot, m, dt, 1000, pad)
        assert sorted_form in (2, 3)
        err = np.abs(got - ref).max() / np.abs(ref).max()
        assert err < (1e-13 if precision == "fp64" else 2e-6), (a, err)


def test_direct_pair_beyond_the_table(torch_cuda):
    torch = torch_cuda
    from paper_1404_7357_gb300 import cfft
    wl = cc.small_patch("fp32", n=1024, n_rho=1024, rho_max=9.0, q_max=4, rotation_classes=1)
    ctx, _ = cc.gpu_table(wl)
    pos = np.array([[0.0, 0.0], [1.0, 0.5], [9.5, 0.0]])
    for block in (0, 1000):
        with pytest.raises(cfft.CfftError):
            _fill(torch, ctx, pos, None, 4, torch.complex64, block)
    _fill(torch, ctx, pos[:2], None, 4, torch.complex64, 0)
