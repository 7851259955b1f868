"""Host logic of batches, without a GPU: the job table and the plan object's bookkeeping (the library
is a fake)."""
import ctypes
from types import SimpleNamespace

import numpy as np
import pytest
import torch

from paper_2106_01326_gb300 import batch
from paper_2106_01326_gb300 import voxtet as vt

STREAM = SimpleNamespace(cuda_stream=0)


class FakeLib:
    """A plan of the library that holds at most ``fit`` jobs in its workspace: wait writes one status
    per job of the last run into the caller's array, if the array holds that many."""

    def __init__(self, fit=8, max_jobs=8):
        self.fit, self.max_jobs, self.n = fit, max_jobs, 0

    def voxtet_default_opts(self, o):
        pass

    def voxtet_plan_create(self, ws, nbytes, max_jobs, opts, handle):
        return vt.OK

    def voxtet_plan_run(self, handle, jobs, n, stream):
        if n > self.max_jobs:
            return vt.ERR_ARG
        self.n = 0
        if n > self.fit:
            return vt.ERR_NOMEM
        self.n = n
        return vt.OK

    def voxtet_plan_wait(self, handle, arr):
        assert len(arr) >= self.n, "statuses written past the array"
        for i in range(self.n):
            arr[i] = vt.ERR_NAN
        return vt.OK

    def voxtet_plan_destroy(self, handle):
        pass


def _specs(n):
    mesh = batch.Mesh(torch.zeros(4, 3), torch.zeros(1, 4, dtype=torch.int32))
    return [batch.JobSpec(mesh, 8, torch.zeros(64, dtype=torch.int32)) for _ in range(n)]


@pytest.fixture()
def plan(monkeypatch):
    lib = FakeLib(fit=4, max_jobs=8)
    monkeypatch.setattr(batch.vt, "load", lambda: lib)
    return batch.Plan(256, 8, device="cpu")


def test_plan_reports_only_runs_that_were_enqueued(plan):
    assert plan.wait() == []
    assert plan.run(_specs(3), stream=STREAM) == vt.OK
    assert plan.wait() == [vt.ERR_NAN] * 3
    assert plan.run(_specs(5), stream=STREAM) == vt.ERR_NOMEM  # does not fit
    assert plan.wait() == []
    assert plan.run(_specs(2), stream=STREAM) == vt.OK
    assert plan.run(_specs(9), stream=STREAM) == vt.ERR_ARG  # refused: the run of two is still the last
    assert plan.wait() == [vt.ERR_NAN] * 2


def test_plan_whose_run_raises_keeps_its_last_run(plan):
    assert plan.run(_specs(4), stream=STREAM) == vt.OK
    bad = _specs(1)
    bad[0].res = None
    with pytest.raises(TypeError):
        plan.run(bad, stream=STREAM)
    assert plan.wait() == [vt.ERR_NAN] * 4


def _origin(value):
    specs = _specs(1)
    specs[0].origin = value
    return list(batch.make_jobs(specs)[0].origin)


@pytest.mark.parametrize("value,want", [
    ((1.0, 2.0, 3.0), [1, 2, 3]),
    ([1, 2, 3], [1, 2, 3]),
    (np.array([1.0, 2.0, 3.0]), [1, 2, 3]),
    (torch.tensor([1.0, 2.0, 3.0]), [1, 2, 3]),
    (1.5, [1.5] * 3),
    (np.float32(1.5), [1.5] * 3),
    ((1.5,), [1.5] * 3),
    (np.array([1.5]), [1.5] * 3),
    (np.array([[1.0, 2.0, 3.0]]), [1, 2, 3]),
], ids=str)
def test_origins_of_a_job(value, want):
    """A job's origin follows numpy's assignment to three float32 values."""
    assert _origin(value) == want


@pytest.mark.parametrize("value", [(1, 2), (1, 2, 3, 4), {1: 0, 2: 0, 3: 0}], ids=str)
def test_origins_that_are_refused(value):
    with pytest.raises((TypeError, ValueError)):
        _origin(value)


def test_one_odd_job_leaves_the_others_alone():
    specs = _specs(5)
    specs[3].origin, specs[4].origin = (0.5,), (1.0, 2.0, 3.0)
    assert [list(j.origin) for j in batch.make_jobs(specs)] == [[0] * 3] * 3 + [[0.5] * 3, [1, 2, 3]]
