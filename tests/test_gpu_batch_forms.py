"""Forms of a batch that only the C entry points give: jobs on lattice coordinates (several prologue
chunks of vertices, one job with a vertex out of range) and a batch that accumulates into its grids.
Against the oracle, as one-off calls and through a plan."""
import ctypes

import numpy as np
import pytest

import oracle
from paper_2106_01326_gb300 import meshgen as mg

pytestmark = pytest.mark.gpu

L = 1 << 20


@pytest.fixture(scope="module")
def env():
    import torch

    if not torch.cuda.is_available():
        pytest.fail("CUDA device required for -m gpu tests")
    from paper_2106_01326_gb300 import batch
    from paper_2106_01326_gb300 import build as vbuild
    from paper_2106_01326_gb300 import voxtet

    vbuild.build()
    oracle.build()
    voxtet.load()
    return voxtet, batch


def _lattice_mesh(n, seed):
    v, t = mg.kuhn_lattice(n, 0.2, seed)
    return np.rint(v.astype(np.float64) * L).astype(np.int32), t.astype(np.int32)


def _run(vt, batch, specs, fixed, plan, accumulate=False):
    """The batch's statuses; ``fixed`` flags the jobs whose vertices are lattice coordinates."""
    import torch

    lib = vt.load()
    jobs = batch.make_jobs(specs)
    for j, f in zip(jobs, fixed):
        j.fixed_point = int(f)
    n = len(specs)
    o = vt.make_opts(0, accumulate, True, not plan)
    nbytes = int(lib.voxtet_batch_workspace_size(jobs, n, n))
    ws = torch.empty(nbytes, dtype=torch.uint8, device="cuda")
    st = (ctypes.c_int32 * n)()
    if not plan:
        assert lib.voxelize_tets_batched(jobs, n, ws.data_ptr(), nbytes, ctypes.byref(o), vt._stream_ptr(None), st) == vt.OK
        return list(st)
    h = ctypes.c_void_p()
    assert lib.voxtet_plan_create(ws.data_ptr(), nbytes, n, ctypes.byref(o), ctypes.byref(h)) == vt.OK
    try:
        for _ in range(2):
            assert lib.voxtet_plan_run(h, jobs, n, vt._stream_ptr(None)) == vt.OK
            assert lib.voxtet_plan_wait(h, st) == vt.OK
    finally:
        lib.voxtet_plan_destroy(h)
    return list(st)


@pytest.mark.parametrize("plan", [False, True], ids=["call", "plan"])
def test_lattice_coordinates(env, plan):
    import torch

    vt, batch = env
    specs, fixed, want, refs = [], [], [], []
    for k, (n, res) in enumerate(((1, 8), (7, 32), (8, 64), (12, 64), (10, 128))):  # 8 to 2,197 vertices: 512 a chunk
        x, t = _lattice_mesh(n, k)
        f = k != 2  # one job in world coordinates among them
        if n == 12:
            x[1000, 1] = 2 * L + 1
        verts = torch.from_numpy(x).cuda() if f else torch.from_numpy((x / L).astype(np.float32)).cuda()
        out = vt.alloc_grid(res)
        out.fill_(-1)
        specs.append(batch.JobSpec(batch.Mesh(verts, torch.from_numpy(t).cuda()), res, out))
        fixed.append(f)
        want.append(vt.ERR_RANGE if n == 12 else vt.OK)
        refs.append(None if n == 12 else oracle.voxelize_fixed(x, t, res))
    assert _run(vt, batch, specs, fixed, plan) == want
    for sp, ref in zip(specs, refs):
        if ref is not None:
            assert np.array_equal(sp.out.cpu().numpy().view(np.uint32).reshape(ref.shape), ref), sp.res


@pytest.mark.parametrize("plan", [False, True], ids=["call", "plan"])
def test_accumulating_batch(env, plan):
    """Every job ORs into what its grid holds; its header and redo bitmap are still cleared."""
    import torch

    vt, batch = env
    rng = np.random.default_rng(4)
    specs, refs = [], []
    for k, (n, res) in enumerate(((3, 32), (9, 64), (5, 128))):
        x, t = _lattice_mesh(n, 20 + k)
        t = t[rng.permutation(len(t))[: len(t) // 3]]
        old = rng.integers(0, 1 << 32, size=vt.grid_words(res), dtype=np.uint64).astype(np.uint32)
        out = torch.from_numpy(old.view(np.int32).copy()).cuda().view(res, res, -1)
        specs.append(batch.JobSpec(batch.Mesh(torch.from_numpy(x).cuda(), torch.from_numpy(np.ascontiguousarray(t)).cuda()), res, out))
        refs.append(oracle.voxelize_fixed(x, t, res).reshape(-1) | old)
    assert _run(vt, batch, specs, [True] * 3, plan, accumulate=True) == [vt.OK] * 3
    for sp, ref in zip(specs, refs):
        assert np.array_equal(sp.out.cpu().numpy().view(np.uint32).reshape(-1), ref), sp.res
