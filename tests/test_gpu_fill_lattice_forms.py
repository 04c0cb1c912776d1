"""The FP64 lattice fill reports itself (fill_form 5) and serves every MBF count of the bucketed
forms (GPU): M = 1, 2 and 4, one and four rotation classes, against the general path (a set row
block, fill_form 2) to the bit; an array that is no lattice, too few elements and missing memory
for the displacements' blocks take the general path."""
import numpy as np
import pytest

import workloads
from tests import cfft_cases as cc

pytestmark = pytest.mark.gpu


def _context(m, classes):
    wl = cc.small_patch("fp64", n=1024, n_rho=1024, rho_max=9.0, q_max=3, rotation_classes=classes)
    wl.element = workloads.patch_rooftops(n_mbf=m)
    return cc.gpu_table(wl)[0]


def _fill(torch, ctx, pos, rot, m, block):
    from paper_1404_7357_gb300 import cfft
    ctx.set_option(cfft.OPT_FILL_BLOCK, block)
    n = len(pos) * m
    z = torch.full((n, n), 7.0, dtype=torch.complex128, device="cuda:0")
    rt = None if rot is None else torch.tensor(rot, device="cuda:0")
    ctx.fill_reduced_matrix(torch.tensor(pos, device="cuda:0"), rt, z)
    return z, ctx.info()["fill_form"]


def _lattice(nx, ny, px, py):
    i, j = np.meshgrid(np.arange(nx), np.arange(ny), indexing="ij")
    return np.stack([i * px, j * py], -1).reshape(-1, 2).astype(float)


@pytest.mark.parametrize("m,classes", [(1, 1), (1, 4), (2, 1), (2, 4), (4, 4)])
def test_form_and_mbf_counts(m, classes):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    ctx = _context(m, classes)
    # pitches of few bits: n coordinates have 2 n - 1 differences
    for pos in (_lattice(18, 18, 0.25, 0.3125), _lattice(11, 29, 0.40625, 0.1875)):
        rot = workloads.rotations(len(pos), seed=31) if classes == 4 else None
        got, form = _fill(torch, ctx, pos, rot, m, 0)
        ref, form_ref = _fill(torch, ctx, pos, rot, m, 1024)
        assert (form, form_ref) == (5, 2)
        assert torch.equal(got, ref)


def test_general_path_is_reported():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1404_7357_gb300 import cfft
    pos = _lattice(18, 18, 0.25, 0.3125)
    ctx = _context(2, 1)
    _, form = _fill(torch, ctx, pos[:250], None, 2, 0)
    assert form == 2
    _, form = _fill(torch, ctx, pos + 1e-3 * np.random.default_rng(1).standard_normal(pos.shape), None, 2, 0)
    assert form == 2
    for after in (0, 1):                                # the coordinates, the blocks
        fresh = _context(2, 1)
        _fill(torch, fresh, pos[:100], None, 2, 0)      # the flags and the fill's own table exist
        cfft.test_fail_allocation(after)
        try:
            got, form = _fill(torch, fresh, pos, None, 2, 0)
        finally:
            cfft.test_fail_allocation(-1)
        ref, _ = _fill(torch, fresh, pos, None, 2, 1024)
        assert form == 2 and torch.equal(got, ref), after
