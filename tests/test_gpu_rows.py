"""The row filter of the slice-unit kernel at its edges, against the oracle, bit for bit.

Structured lattices put sample rows exactly on faces; where every face's row bound is a multiple of
1/16 sample the filter must decide those ties itself (no row is left to the exact kernels).
"""
import numpy as np
import pytest

import oracle
from paper_2106_01326_gb300 import meshgen as mg

pytestmark = pytest.mark.gpu

L = 1 << 20


@pytest.fixture(scope="module")
def vt():
    import torch

    if not torch.cuda.is_available():
        pytest.fail("CUDA device required for -m gpu tests")
    from paper_2106_01326_gb300 import build as vbuild
    from paper_2106_01326_gb300 import voxtet

    vbuild.build()
    oracle.build()
    voxtet.load()
    return voxtet


def run_fixed(vt, xyz, tets, res, **kw):
    import torch

    t = torch.from_numpy(np.ascontiguousarray(tets, dtype=np.int32)).cuda()
    x = torch.from_numpy(np.ascontiguousarray(xyz, dtype=np.int32)).cuda()
    ws = vt.alloc_workspace(len(tets), len(xyz), res)
    g = vt.voxelize_fixed(x, t, res, workspace=ws, **kw)
    return g.cpu().numpy().view(np.uint32), vt.read_stats(ws)


@pytest.mark.parametrize("mode", [0, 1])
@pytest.mark.parametrize("n,res,half", [(1, 8, 0), (4, 16, 1), (8, 64, 1), (16, 64, 0), (8, 128, 1), (3, 64, 1), (6, 32, 0)])
def test_lattice_ties_are_certified(vt, n, res, half, mode):
    """Kuhn lattices moved by whole voxels plus `half` a voxel: faces x = y, y = z, x = const through
    sample centres.  With a power-of-two lattice every row bound is a multiple of 1/2, so no row may be
    queued by the slice-unit kernel (tets of at most 16 slices); the others only have to give the
    oracle's grid."""
    ijk, tets = mg.kuhn_lattice_int(n)
    step = L // res
    xyz = ijk * (L // n) + np.array([1, -2, 3]) * step + half * (step // 2)
    got, st = run_fixed(vt, xyz, tets, res, mode=mode, kernel=2)
    ref = oracle.voxelize_fixed(xyz.astype(np.int32), tets, res, mode=mode)
    assert np.array_equal(got.reshape(ref.shape), ref)
    if n & (n - 1) == 0 and res // n < 16:
        assert st["fallback_rows"] == 0, st


@pytest.mark.parametrize("mode", [0, 1])
def test_faces_just_off_a_sixteenth(vt, mode):
    """Tets whose face x = y is off by one lattice unit in one vertex: the slope is within the look of a
    multiple of 1/16 but is none, so the exact check must refuse it and ties elsewhere stay right."""
    rng = np.random.default_rng(5)
    res = 32
    step = L // res
    xyz, tets = [], []
    for k in range(400):
        o = (rng.integers(2, 26, size=3) * 2 + 1) * (step // 2)
        s = int(rng.integers(1, 5)) * step
        v = np.array([[0, 0, 0], [s, s, 0], [s, s, s], [s, 0, 0]]) + o
        v[int(rng.integers(4)), int(rng.integers(3))] += int(rng.integers(-1, 2))
        tets.append(np.arange(4) + 4 * k)
        xyz.append(v)
    xyz, tets = np.concatenate(xyz).astype(np.int32), np.array(tets, dtype=np.int32)
    got, _ = run_fixed(vt, xyz, tets, res, mode=mode, kernel=2)
    ref = oracle.voxelize_fixed(xyz, tets, res, mode=mode)
    assert np.array_equal(got.reshape(ref.shape), ref)
