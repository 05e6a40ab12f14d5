"""Solver.solve on device tensors: the copy that turns U into columns is enqueued on the caller's stream, so the
handle's stream has to wait for that stream after the copy and before the solve. Read from the order of the calls, on
the CPU, with the streams and the library call replaced by recorders."""
import pytest

torch = pytest.importorskip("torch")


class Recorder:
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
