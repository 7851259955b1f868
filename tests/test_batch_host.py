"""Host logic of batches, without a GPU: the plan object's bookkeeping (the library is a fake)."""
import ctypes
from types import SimpleNamespace

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
