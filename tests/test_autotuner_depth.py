"""The batch autotuner and the depth that mf_zchunk = 0 stands for (2 node
planes on small cells, 8 on large ones), with a fake solver on the host: the
depth a handle runs at is the one that was timed fastest, the small cells' own
depth is among the candidates, and a shape that was not searched keeps the
library's depth, also across cache files."""
import contextlib
import json
import types

import pytest
import torch

from paper_2602_07225_gb300 import batch
from paper_2602_07225_gb300.batch import SETUP_CANDIDATES, SETUP_DEFAULT, Autotuner, BatchSolver

CASE = {"mesh": {"nx": 16, "ny": 16, "nz": 24}, "state": None}
KEY = (16, 16, 24, 1)


class FakeSolver:
    """A small cell: the time of a solve by the depth in use."""
    ms = {}

    def __init__(self, case, device=None, stream=None, coarse_max=128, mf_zchunk=0, **opts):
        self.stream = stream
        self.params = types.SimpleNamespace(precision=1, coarse_max=coarse_max, mf_zchunk=mf_zchunk)

    def running(self):
        return (self.params.coarse_max, self.params.mf_zchunk or 2)

    def state_tensors(self, st):
        return None

    def residual(self, st):
        return torch.zeros(1)

    def jacobian_update(self, st):
        pass

    def set_options(self, **o):
        pass

    def solve(self, b, check=True):
        return None, {"status": 0, "ms_total": self.ms.get(self.running(), 9.0)}

    def close(self):
        pass


@pytest.fixture(autouse=True)
def _host(monkeypatch):
    monkeypatch.setattr(batch, "P4DSolver", FakeSolver)
    monkeypatch.setattr(torch.cuda, "Stream", lambda device=None: None)
    monkeypatch.setattr(torch.cuda, "stream", lambda s: contextlib.nullcontext())
    monkeypatch.setattr(torch.cuda, "synchronize", lambda *a: None)


@pytest.mark.parametrize("best", [(128, 8), (128, 2), (128, 4), (64, 8)])
def test_handle_runs_at_the_depth_that_was_fastest(monkeypatch, best):
    # the next fastest is 4 planes
    monkeypatch.setattr(FakeSolver, "ms", {(128, 4): 3.0, best: 1.0})
    bs = BatchSolver([CASE, CASE], tune_setup=True)
    assert best in SETUP_CANDIDATES and bs.tuned[KEY][4:] == best
    assert [s.running() for s in bs.solvers] == [best, best]


def test_shape_without_a_search_keeps_the_librarys_depth_until_one_runs(monkeypatch, tmp_path):
    monkeypatch.setattr(FakeSolver, "ms", {(128, 8): 1.0, (128, 2): 2.0})
    path = str(tmp_path / "t.json")
    bs = BatchSolver([CASE], tuner=Autotuner(path))
    assert bs.tuned[KEY][4:] == SETUP_DEFAULT and bs.solvers[0].running() == (128, 2)
    bs = BatchSolver([CASE], tuner=Autotuner(path), tune_setup=True)       # the file held no search
    assert bs.solvers[0].running() == (128, 8)
    bs = BatchSolver([CASE], tuner=Autotuner(path))                        # now it does
    assert bs.tuned[KEY][4:] == (128, 8) and bs.solvers[0].running() == (128, 8)


def test_older_file_gives_the_runtime_options_only(monkeypatch, tmp_path):
    monkeypatch.setattr(FakeSolver, "ms", {(128, 2): 1.0})
    path = str(tmp_path / "old.json")
    json.dump({json.dumps(list(KEY)): [3, 20.0, 0, [1, 0, 2], 128, 4]}, open(path, "w"))
    bs = BatchSolver([CASE], tuner=Autotuner(path))
    assert bs.tuned[KEY][:2] == (3, 20.0) and bs.solvers[0].running() == (128, 2)
    bs = BatchSolver([CASE], tuner=Autotuner(path), tune_setup=True)
    assert bs.tuned[KEY] == (3, 20.0, 0, [1, 0, 2], 128, 2) and bs.solvers[0].running() == (128, 2)
