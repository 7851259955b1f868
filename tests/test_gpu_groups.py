"""Slice units shared by groups of threads, taken in windows, listed per slab and batched: where a tet's
slices and rows exceed one window, and where few or wide tets are shared by many threads.  All bit for
bit against the oracle."""
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


def _cuda(verts, tets):
    import torch

    return torch.from_numpy(np.ascontiguousarray(verts)).cuda(), torch.from_numpy(np.ascontiguousarray(tets)).cuda()


def _soup(seed, n, res, lo, hi, axis_scale=(1.0, 1.0, 1.0)):
    """n tets of lo..hi voxels (times axis_scale) anywhere in the unit cube, some flat or inverted."""
    rng = np.random.default_rng(seed)
    o = rng.random((n, 1, 3))
    size = np.exp(rng.uniform(np.log(lo), np.log(hi), size=(n, 1, 1))) / res * np.asarray(axis_scale)
    v = (o + (rng.random((n, 4, 3)) - 0.5) * size).astype(np.float32)
    v[8::17, 3] = v[8::17, 2]  # zero volume
    return v.reshape(-1, 3), np.arange(4 * n, dtype=np.int32).reshape(n, 4)


def _same(got, ref, what):
    got = got.cpu().numpy().view(np.uint32)
    assert np.array_equal(got.reshape(ref.shape), ref), what


@pytest.mark.parametrize("mode", [0, 1])
@pytest.mark.parametrize("n,res,lo,hi", [(1, 128, 90, 120), (3, 256, 60, 200), (40, 128, 1, 100), (700, 64, 1, 60),
                                         (5000, 128, 1, 8), (20000, 64, 0.5, 20), (140000, 32, 0.3, 3)])
def test_groups_and_windows(vt, n, res, lo, hi, mode):
    """From one tet (a whole block shares it) to meshes with a thread a tet, in both cases with tets of
    more slices than a window holds."""
    verts, tets = _soup(n, n, res, lo, hi)
    ref = oracle.voxelize(verts, tets, (0, 0, 0), 1.0 / res, res, mode=mode)
    v, t = _cuda(verts, tets)
    _same(vt.voxelize(v, t, (0, 0, 0), 1.0 / res, res, mode=mode), ref, "culled")
    _same(vt.voxelize(v, t, (0, 0, 0), 1.0 / res, res, mode=mode, row_cull=2), ref, "all rows")


@pytest.mark.parametrize("dims,scale", [((40, 2100, 24), (0.2, 2, 0.2)), ((17, 1030, 9), (0.3, 2.1, 0.3)),
                                        ((5000, 20, 12), (2, 0.3, 0.3)), ((9, 12, 1200), (0.3, 0.3, 2))])
def test_more_rows_and_columns_than_a_window(vt, dims, scale):
    """Boxes of more than 1024 rows per slice, of thousands of columns, and of 1200 slices."""
    h = 1.0 / 64
    verts, tets = _soup(3, 300, 64, 4, 30, scale)
    verts = verts * np.array([dims[0] * h, dims[1] * h, dims[2] * h], dtype=np.float32)
    ref = oracle.voxelize_grid(verts, tets, (0, 0, 0), h, dims)
    v, t = _cuda(verts, tets)
    _same(vt.voxelize_grid(v, t, (0, 0, 0), h, dims), ref, dims)


@pytest.mark.parametrize("z0,z1", [(0, 1), (31, 33), (40, 52), (99, 100), (60, 72)])
@pytest.mark.parametrize("n,lo,hi", [(50, 5, 90), (9000, 1, 6)])
def test_thin_slab_lists(vt, n, lo, hi, z0, z1):
    """Slabs below an eighth of the grid go through the list of their tets; tets wider than the exact
    integers of the filter path go to the exact kernel from there, flat ones are only counted."""
    dims, h = (90, 70, 100), 1.0 / 128
    verts, tets = _soup(n, n, 128, lo, hi)
    wide = np.array([[-0.9, -0.9, -0.5], [1.9, 0.1, 0.4], [0.2, 1.9, 0.6], [0.3, 0.4, 1.7]], dtype=np.float32)
    tets = np.concatenate([tets, [[len(verts) + k for k in range(4)]]]).astype(np.int32)
    verts = np.concatenate([verts, wide])
    ref = oracle.voxelize_grid(verts, tets, (0, 0, 0), h, dims, z0=z0, z1=z1)
    v, t = _cuda(verts, tets)
    ws = vt.alloc_workspace(len(tets), len(verts), 100)
    _same(vt.voxelize_grid(v, t, (0, 0, 0), h, dims, z_range=(z0, z1), workspace=ws), ref, (z0, z1))
    st = vt.read_stats(ws)
    assert st["wide_tets"] == 1 and st["degenerate_tets"] >= len(range(8, n, 17))
    bad = tets.copy()
    bad[len(bad) // 2, 1] = len(verts)
    st, _ = vt.voxelize_grid(v, _cuda(verts, bad)[1], (0, 0, 0), h, dims, z_range=(z0, z1), raise_on_error=False)
    assert st == vt.ERR_INDEX


@pytest.mark.parametrize("n,res", [(4, 256), (6, 256)])
@pytest.mark.parametrize("mode", [0, 1])
def test_wide_tets_few_rows_left_to_the_exact_kernels(vt, n, res, mode):
    """Tets of 43 and 64 voxels: a steep face's error would give up most of a tet's rows if it stood
    for the whole side; with each face's own error few are left."""
    verts, tets = mg.kuhn_lattice(n, jitter=0.25, seed=11)
    verts, tets = verts.astype(np.float32), tets.astype(np.int32)
    ref = oracle.voxelize(verts, tets, (0, 0, 0), 1.0 / res, res, mode=mode)
    v, t = _cuda(verts, tets)
    ws = vt.alloc_workspace(len(tets), len(verts), res)
    _same(vt.voxelize(v, t, (0, 0, 0), 1.0 / res, res, mode=mode, workspace=ws), ref, (n, res))
    st = vt.read_stats(ws)
    assert st["fallback_rows"] < 0.01 * st["rows"], st


@pytest.mark.parametrize("use_filter", [True, False])
def test_batch_of_unlike_jobs(vt, use_filter):
    """One batch with jobs of one tet, of wide tets, of many small ones, without tets, in lattice
    coordinates and with an unaligned grid; each job's grid and status are its own."""
    import torch

    from paper_2106_01326_gb300 import batch

    specs, refs = [], []
    store = torch.full((1 << 20,), -1, dtype=torch.int32, device="cuda")
    at = 1  # grids start on 4-byte boundaries only
    for seed, n, res, lo, hi in ((1, 1, 64, 30, 60), (2, 300, 128, 10, 120), (3, 30000, 32, 0.3, 4), (4, 0, 64, 1, 2),
                                 (5, 900, 64, 1, 50), (6, 129, 1, 0.5, 1), (7, 4000, 128, 1, 9)):
        verts, tets = _soup(seed, n, res, lo, hi) if n else (np.zeros((0, 3), np.float32), np.zeros((0, 4), np.int32))
        v, t = _cuda(verts, tets)
        w = vt.grid_words(res)
        specs.append(batch.JobSpec(batch.Mesh(v, t), res, store[at:at + w].view(res, res, -1)))
        at += w
        refs.append(oracle.voxelize(verts, tets, (0, 0, 0), 1.0 / res, res) if n else np.zeros((res, res, (res + 31) // 32), np.uint32))
    # a tet wider than the filter path's integers: the batch's exact kernel takes it
    wide = np.array([[-0.9, -0.9, -0.5], [1.9, 0.1, 0.4], [0.2, 1.9, 0.6], [0.3, 0.4, 1.7]], dtype=np.float32)
    v, t = _cuda(wide, np.arange(4, dtype=np.int32).reshape(1, 4))
    specs.append(batch.JobSpec(batch.Mesh(v, t), 32, store[at:at + vt.grid_words(32)].view(32, 32, -1)))
    at += vt.grid_words(32)
    refs.append(oracle.voxelize(wide, np.arange(4, dtype=np.int32).reshape(1, 4), (0, 0, 0), 1.0 / 32, 32))
    bad = _soup(8, 60, 64, 1, 9)
    bad_v = bad[0].copy()
    bad_v[7, 1] = np.nan
    v, t = _cuda(bad_v, bad[1])
    specs.append(batch.JobSpec(batch.Mesh(v, t), 64, store[at:at + vt.grid_words(64)].view(64, 64, -1)))
    for _ in range(2):
        assert batch.voxelize_batched(specs, use_filter=use_filter) == [vt.OK] * len(refs) + [vt.ERR_NAN]
        for k, (sp, ref) in enumerate(zip(specs, refs)):
            _same(sp.out, ref, k)
    assert int(store[0]) == -1 and int(store[at + vt.grid_words(64)]) == -1


@pytest.mark.parametrize("rx,shift", [(640, 0), (640, 1), (608, 0), (609, 0), (1000, 0), (1000, 3), (700, 2)])
@pytest.mark.parametrize("mode", [0, 1])
def test_rows_in_pairs_of_words(vt, rx, shift, mode):
    """Grids above 512 per side: rows of even and odd numbers of words in grids that start on 8-byte and
    on 4-byte boundaries, tets of 1 to 400 columns (rows of one pair, two, and whole pairs between)."""
    import torch

    dims, h = (rx, 24, 18), 1.0 / 1024
    verts, tets = _soup(rx, 400, 24, 2, 24, (0.6, 1, 1))
    verts = verts * np.array([dims[0] * h, dims[1] * h, dims[2] * h], dtype=np.float32)
    ref = oracle.voxelize_grid(verts, tets, (0, 0, 0), h, dims, mode=mode)
    v, t = _cuda(verts, tets)
    w = (rx + 31) // 32
    store = torch.full((dims[1] * dims[2] * w + 8,), -1, dtype=torch.int32, device="cuda")
    out = store[shift:shift + dims[1] * dims[2] * w].view(dims[2], dims[1], w)
    _same(vt.voxelize_grid(v, t, (0, 0, 0), h, dims, out=out, mode=mode), ref, (rx, shift))
    assert bool((store[:shift] == -1).all()) and bool((store[shift + ref.size:] == -1).all())


def _wide_among_small(seed, n, res, wide, lo, hi, where, axis_scale=(1.0, 1.0, 1.0)):
    """n tets of a few voxels with `wide` of lo..hi voxels: at the end, the start, or spread."""
    small, t0 = _soup(seed, n, res, 0.5, 3)
    big, t1 = _soup(seed + 1, wide, res, lo, hi, axis_scale)
    tets = np.concatenate([t0, t1 + len(small)]).astype(np.int32)
    if where == "start":
        tets = np.roll(tets, wide, axis=0)
    elif where == "spread":
        tets = tets[np.random.default_rng(seed).permutation(len(tets))]
    return np.concatenate([small, big]), np.ascontiguousarray(tets)


@pytest.mark.parametrize("where", ["end", "start", "spread"])
@pytest.mark.parametrize("n,wide,res,lo,hi", [(120000, 1, 64, 50, 64), (120000, 20, 64, 20, 64), (9000, 300, 64, 15, 40),
                                              (9000, 65, 128, 60, 128), (300, 127, 128, 33, 100)])
def test_wide_tets_among_small_ones(vt, n, wide, res, lo, hi, where):
    """Only the tets with slices left go on to a tile's next window, shared by more threads: from one
    tet of a tile to nearly all of them, several windows deep."""
    verts, tets = _wide_among_small(n + wide, n, res, wide, lo, hi, where)
    ref = oracle.voxelize(verts, tets, (0, 0, 0), 1.0 / res, res)
    v, t = _cuda(verts, tets)
    ws = vt.alloc_workspace(len(tets), len(verts), res)
    got = vt.voxelize(v, t, (0, 0, 0), 1.0 / res, res, workspace=ws)
    _same(got, ref, "one call")
    flat = len(range(8, n, 17)) + len(range(8, wide, 17))
    assert vt.read_stats(ws)["degenerate_tets"] >= flat  # each counted once, in its first window
    _same(vt.voxelize(v, t, (0, 0, 0), 1.0 / res, res, row_cull=2, mode=0), ref, "all rows")
    from paper_2106_01326_gb300 import batch

    specs = [batch.JobSpec(batch.Mesh(v, t), res, vt.alloc_grid(res)) for _ in range(3)]
    assert batch.voxelize_batched(specs) == [vt.OK] * 3
    for sp in specs:
        _same(sp.out, ref, "batch")


@pytest.mark.parametrize("dims,scale,lo,hi", [((24, 2600, 40), (0.3, 1, 0.3), 300, 2600), ((24, 1500, 150), (0.2, 1, 1), 60, 1500),
                                              ((600, 30, 300), (1, 0.2, 1), 40, 300)])
@pytest.mark.parametrize("z", [None, (3, 8)])
def test_tall_tets_among_small_ones(vt, dims, scale, lo, hi, z):
    """Tets of more than 1024 rows, with and without more slices than a window holds, among small ones,
    in whole grids and in slabs listed first."""
    h = 1.0 / 4096
    verts, tets = _wide_among_small(dims[1], 3000, max(dims), 30, lo, hi, "spread", scale)
    verts = (verts * np.array([d * h for d in dims])).astype(np.float32)
    z0, z1 = z or (0, dims[2])
    ref = oracle.voxelize_grid(verts, tets, (0, 0, 0), h, dims, z0=z0, z1=z1)
    v, t = _cuda(verts, tets)
    for mode_cull in (0, 2):
        _same(vt.voxelize_grid(v, t, (0, 0, 0), h, dims, z_range=(z0, z1), row_cull=mode_cull), ref, (dims, z, mode_cull))


@pytest.mark.parametrize("z0,z1", [(300, 325), (400, 410)])
def test_slab_of_long_thin_tets(vt, z0, z1):
    """A slab's listed tets of 25 and 10 slices and a few rows each, shared by as many threads as hold
    their slices in one window."""
    dims, h = (30, 24, 900), 1.0 / 1024
    verts, tets = _soup(77, 4000, 900, 20, 300, (0.01, 0.01, 1.0))
    verts = (verts * np.array([d * h for d in dims])).astype(np.float32)
    ref = oracle.voxelize_grid(verts, tets, (0, 0, 0), h, dims, z0=z0, z1=z1)
    v, t = _cuda(verts, tets)
    _same(vt.voxelize_grid(v, t, (0, 0, 0), h, dims, z_range=(z0, z1)), ref, (z0, z1))


@pytest.mark.parametrize("n,dims,lo,hi,scale", [(1, (40, 2100, 48), 30, 60, (0.3, 1, 1)), (5, (700, 300, 48), 10, 60, (1, 1, 1)),
                                                (300, (64, 64, 64), 5, 60, (1, 1, 1)), (5000, (64, 64, 64), 1, 20, (1, 1, 1)),
                                                (270000, (64, 64, 64), 0.3, 2, (1, 1, 1)), (40, (24, 20, 900), 30, 300, (0.1, 0.1, 1))])
@pytest.mark.parametrize("nz", [1, 2, 4, 5, 7])
def test_slabs_of_a_few_slices(vt, n, dims, lo, hi, scale, nz):
    """Up to four slices of a small mesh go without a list, in tiles of fewer tets where those are few;
    thicker slabs and larger meshes through a list."""
    h = 1.0 / 4096
    verts, tets = _soup(n, n, max(dims[2], 48), lo, hi, scale)
    verts = (verts * np.array([d * h for d in dims])).astype(np.float32)
    z0 = dims[2] // 2 - 1
    ref = oracle.voxelize_grid(verts, tets, (0, 0, 0), h, dims, z0=z0, z1=z0 + nz)
    v, t = _cuda(verts, tets)
    for mode_cull in (0, 2):
        got = vt.voxelize_grid(v, t, (0, 0, 0), h, dims, z_range=(z0, z0 + nz), row_cull=mode_cull)
        _same(got, ref, (n, dims, nz, mode_cull))
