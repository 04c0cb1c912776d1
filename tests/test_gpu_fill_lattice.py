"""The FP64 fill of arrays whose pairs repeat their displacements (GPU).

Arrays of at least 256 elements on few coordinate values evaluate each displacement once and
copy the blocks; a set row block (option FILL_BLOCK) keeps the general path.  Both see the same
differences of coordinates, so the matrices are equal to the bit: square, rectangular, offset
and incomplete lattices in any element order, one and four rotation classes, a padded leading
dimension, and an array with displacements beyond the table that no pair has.
"""
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


def _lattice(nx, ny, px, py, shift=0.0):
    i, j = np.meshgrid(np.arange(nx), np.arange(ny), indexing="ij")
    return np.stack([i * px + (j % 2) * shift, j * py], -1).reshape(-1, 2)


def _cross(n, thick, pitch):
    i, j = np.meshgrid(np.arange(n), np.arange(n), indexing="ij")
    lo, hi = (n - thick) // 2, (n + thick) // 2
    keep = ((i >= lo) & (i < hi)) | ((j >= lo) & (j < hi))
    return pitch * np.stack([i[keep], j[keep]], -1).astype(float)


def _arrays():
    rng = np.random.default_rng(5)
    square = _lattice(17, 17, 0.3517, 0.3517)
    holes = _lattice(20, 20, 0.25, 0.25)
    return {"square": square,
            "rectangle": _lattice(10, 30, 0.41, 0.173),
            "offset": _lattice(18, 18, 0.25, 0.25, shift=0.125),
            "holes": holes[rng.permutation(len(holes))[:330]],
            "cross": _cross(32, 8, 0.25),          # its bounding box's diagonal is beyond the table
            "row": _lattice(90, 3, 0.0625, 0.5)}


def _fill(torch, ctx, pos, rot, m, block, pad):
    from paper_1404_7357_gb300 import cfft
    a = len(pos)
    ctx.set_option(cfft.OPT_FILL_BLOCK, block)
    z = torch.full((a * m, a * m + pad), 7.0, dtype=torch.complex128, device="cuda:0")
    rt = None if rot is None else torch.tensor(rot, device="cuda:0")
    ctx.fill_reduced_matrix(torch.tensor(pos, device="cuda:0"), rt, z)
    return z


@pytest.mark.parametrize("classes", [1, 4])
def test_lattice_matches_general_path(torch_cuda, classes):
    torch = torch_cuda
    wl = cc.small_patch("fp64", n=1024, n_rho=1024, rho_max=9.0, q_max=4, rotation_classes=classes)
    ctx, _ = cc.gpu_table(wl)
    for name, pos in _arrays().items():
        pos = pos[np.random.default_rng(9).permutation(len(pos))]
        rot = workloads.rotations(len(pos), seed=31) if classes == 4 else None
        pad = 3 if name == "square" else 0
        got = _fill(torch, ctx, pos, rot, 4, 0, pad)
        ref = _fill(torch, ctx, pos, rot, 4, 1024, pad)
        assert torch.equal(got, ref), name


def test_lattice_pair_beyond_the_table(torch_cuda):
    torch = torch_cuda
    from paper_1404_7357_gb300 import cfft
    wl = cc.small_patch("fp64", n=1024, n_rho=1024, rho_max=9.0, q_max=4, rotation_classes=1)
    ctx, _ = cc.gpu_table(wl)
    for block in (0, 1024):
        with pytest.raises(cfft.CfftError):
            _fill(torch, ctx, _cross(32, 8, 0.3125), None, 4, block, 0)
    ok = _cross(32, 8, 0.25)
    assert torch.equal(_fill(torch, ctx, ok, None, 4, 0, 0), _fill(torch, ctx, ok, None, 4, 1024, 0))
