"""The handle's stream waits for the caller's after what the caller's stream still has to do for the call: the copy that
turns U into columns (Solver.solve on device tensors), and whatever used the workspace's memory before (Solver). Read
from the order of the calls, on the CPU, with the streams and the library calls replaced by recorders."""
import pytest

import workloads as wl

torch = pytest.importorskip("torch")


class Recorder:
    cuda_stream = 0

    def __init__(self, log):
        self.log = log

    def wait_stream(self, other):
        self.log.append("wait")


class DeviceVector:
    is_cuda = True
    device = torch.device("cpu")


class Block:
    def __init__(self, log, dims):
        self.log, self.dims = log, dims

    def dim(self):
        return self.dims

    def t(self):
        return self

    def contiguous(self):
        self.log.append("copy of U")
        return self


@pytest.mark.parametrize("dims", [None, 1, 2])
def test_the_handle_waits_for_the_copy_of_u(monkeypatch, dims):
    import paper_2608_07327_gb300 as mb
    log = []
    sv = object.__new__(mb.Solver)
    sv.n, sv.h, sv.stream = 5, None, Recorder(log)
    monkeypatch.setattr(torch.cuda, "current_stream", lambda *a: None)

    def solve_dev(h, b, U, tol, maxit, x):
        log.append("solve")
        return mb.MBPCG_OK, mb.Info()

    monkeypatch.setattr(mb, "mbpcg_solve_dev", solve_dev)
    sv.solve(DeviceVector(), None if dims is None else Block(log, dims))
    assert log == (["copy of U"] if dims == 2 else []) + ["wait", "solve"]


@pytest.mark.parametrize("dense", [False, True])
def test_the_handle_waits_for_the_memory_of_its_workspace(monkeypatch, dense):
    import paper_2608_07327_gb300 as mb
    log = []
    monkeypatch.setattr(torch.cuda, "is_available", lambda: True)
    monkeypatch.setattr(torch.cuda, "Stream", lambda: Recorder(log))
    monkeypatch.setattr(torch.cuda, "current_stream", lambda *a: None)
    monkeypatch.setattr(torch, "empty", lambda *a, **k: log.append("workspace"))
    for kind in ("csr", "dense"):
        monkeypatch.setattr(mb, "mbpcg_workspace_size_" + kind, lambda *a: 256)
        monkeypatch.setattr(mb, "mbpcg_create_" + kind, lambda *a: log.append("create"))
    mb.Solver(wl.dense_mtm(4, 1) if dense else wl.poisson2d(3))
    assert log == ["workspace", "wait", "create"]
