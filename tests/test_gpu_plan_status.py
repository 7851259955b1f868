"""Statuses of a batch plan: each replay reports its own jobs' errors at their places, and a run
that failed leaves nothing to read (no status of an earlier, larger batch)."""
import ctypes

import numpy as np
import pytest

from paper_2106_01326_gb300 import meshgen as mg

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    import torch

    if not torch.cuda.is_available():
        pytest.fail("CUDA device required for -m gpu tests")
    from paper_2106_01326_gb300 import batch
    from paper_2106_01326_gb300 import build as vbuild
    from paper_2106_01326_gb300 import voxtet

    vbuild.build()
    voxtet.load()
    return voxtet, batch


def _job(vt, batch, n=4, res=32, spoil=None):
    v, t = mg.kuhn_lattice(n, 0.2, 5)
    if spoil == "nan":
        v = v.copy()
        v[7, 2] = np.nan
    elif spoil == "index":
        t = t.copy()
        t[3, 1] = len(v)
    elif spoil == "range":
        v = v.copy()
        v[2, 0] = 9.0
    return batch.JobSpec(batch.Mesh.from_numpy(v, t), res, vt.alloc_grid(8 if res == 12 else res))


def test_replays_report_their_own_errors(env):
    vt, batch = env
    codes = {"nan": vt.ERR_NAN, "index": vt.ERR_INDEX, "range": vt.ERR_RANGE, "res": vt.ERR_RES, None: vt.OK}
    kinds = [["nan", None, "res", None, "index", None, None, "range"],
             [None] * 5,
             [None, "index", None],
             [None, None, "range", "nan", "res", None, None, None],
             [None] * 8]
    batches = [[_job(vt, batch, 3 + i % 3, 12 if k == "res" else 32, None if k == "res" else k)
                for i, k in enumerate(ks)] for ks in kinds]
    plan = batch.Plan(max(batch.batch_workspace_size(b, 8) for b in batches), 8)
    try:
        for ks, specs in list(zip(kinds, batches)) * 2:
            assert plan.run(specs) == vt.OK
            assert plan.wait() == [codes[k] for k in ks]
            assert plan.wait() == [codes[k] for k in ks]  # asked again
    finally:
        plan.close()


def test_failed_run_leaves_no_statuses(env):
    """The C entry points: eight jobs run, then one that does not fit, then two that do."""
    vt, batch = env
    lib = vt.load()
    good = [_job(vt, batch) for _ in range(8)]
    plan = batch.Plan(batch.batch_workspace_size(good, 8), 8)
    big = batch.JobSpec(good[0].mesh, 32, good[0].out)
    table = batch.make_jobs([big])
    table[0].n_tets = 50_000_000  # a workspace far beyond the plan's; refused before anything is read
    stream = vt._stream_ptr(None)
    try:
        assert plan.run(good) == vt.OK
        assert plan.wait() == [vt.OK] * 8
        assert lib.voxtet_plan_run(plan._handle, table, 1, stream) == vt.ERR_NOMEM
        seen = (ctypes.c_int32 * 8)(*[77] * 8)
        assert lib.voxtet_plan_wait(plan._handle, seen) == vt.OK
        assert list(seen) == [77] * 8
        jobs = batch.make_jobs(good[:2])
        assert lib.voxtet_plan_run(plan._handle, jobs, 2, stream) == vt.OK
        assert lib.voxtet_plan_run(plan._handle, jobs, 9, stream) == vt.ERR_ARG  # more than the plan holds
        assert lib.voxtet_plan_wait(plan._handle, seen) == vt.OK
        assert list(seen) == [vt.OK] * 2 + [77] * 6
    finally:
        plan.close()
