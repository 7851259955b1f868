"""The exact kernel's whole-tet path, bit for bit against the oracle: 64-bit and 128-bit tets in turn
through the same blocks (their face data shares one place in shared memory), with every number of
upper, lower and x-parallel faces, and boxes of a few rows to many times the block's threads."""
import numpy as np
import pytest

import oracle

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


def mixed_tets(seed, n, wide):
    """n tets in lattice units; the share ``wide`` of them extends past 2^20 (up to the coordinate
    limit).  Half of the tets are on a coarse lattice: faces parallel to the axes, exact ties."""
    rng = np.random.default_rng(seed)
    size = np.exp(rng.uniform(np.log(L / 200), np.log(0.9 * L), (n, 1, 1)))
    x = rng.uniform(0, L, (n, 1, 3)) + size * rng.uniform(-0.5, 0.5, (n, 4, 3))
    big = rng.random(n) < wide
    x[big] = rng.uniform(-2 * L, 2 * L, (int(big.sum()), 4, 3))
    x[big, 0] = rng.uniform(0, L, (int(big.sum()), 3))
    coarse = rng.random(n) < 0.5
    x[coarse] = np.round(x[coarse] / (L // 32)) * (L // 32)
    x = np.clip(np.rint(x), -2 * L, 2 * L).astype(np.int32)
    return x.reshape(-1, 3), np.arange(4 * n, dtype=np.int32).reshape(n, 4)


@pytest.mark.parametrize("mode", [0, 1])
@pytest.mark.parametrize("n,wide,res", [(1, 1.0, 64), (1, 0.0, 64), (900, 0.3, 32), (2500, 0.02, 64), (300, 0.5, 128)])
def test_mixed_widths(vt, n, wide, res, mode):
    import torch

    xyz, tets = mixed_tets(n + mode, n, wide)
    if n == 1:
        xyz = np.array([[0, 0, 0], [2 * L if wide else L, 0, 0], [0, L, 0], [0, 0, L]], dtype=np.int32)
    ref = oracle.voxelize_fixed(xyz, tets, res, mode=mode)
    x, t = torch.from_numpy(xyz).cuda(), torch.from_numpy(tets).cuda()
    ws = vt.alloc_workspace(len(tets), len(xyz), res)
    for use_filter in (False, True):
        got = vt.voxelize_fixed(x, t, res, mode=mode, use_filter=use_filter, workspace=ws)
        assert np.array_equal(got.cpu().numpy().view(np.uint32).reshape(ref.shape), ref), use_filter
        st = vt.read_stats(ws)
        assert st["wide_tets"] == 0 or wide > 0
        if not use_filter:
            assert st["exact_tets"] > 0.4 * n


@pytest.mark.parametrize("kernel", [1, 2], ids=["spans", "slices"])
@pytest.mark.parametrize("n,res", [(4, 32), (6, 128), (12, 128)])
def test_rows_queued_past_a_blocks_stage(vt, n, res, kernel):
    """Cells of 4:12:12, whose faces meet sample centres every third row: each tile queues many times the
    rows a block stages (512 in the span kernel, 64 in the slice-unit kernel), the largest mesh more
    than the row queue holds, so that whole tets are solved again."""
    import torch

    from paper_2106_01326_gb300 import meshgen as mg

    ijk, tets = mg.kuhn_lattice_int(n)
    half = L // 2 // res
    unit = max(1, L // (12 * n) // (2 * half // 8)) * (2 * half // 8)
    xyz = (ijk * (np.array([4, 12, 12]) * unit) + half).astype(np.int32)
    ref = oracle.voxelize_fixed(xyz, tets, res)
    x, t = torch.from_numpy(xyz).cuda(), torch.from_numpy(tets).cuda()
    ws = vt.alloc_workspace(len(tets), len(xyz), res)
    got = vt.voxelize_fixed(x, t, res, workspace=ws, kernel=kernel)
    assert np.array_equal(got.cpu().numpy().view(np.uint32).reshape(ref.shape), ref)
    queued = vt.read_stats(ws)["fallback_rows"]
    assert queued > 512 and (n < 12 or queued > 65536)
