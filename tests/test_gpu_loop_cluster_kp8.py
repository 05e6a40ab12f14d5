"""The one-cluster loop at padded width 8, whose k x k steps run on two warps: both have to take the same
decision on every pivot, in every CTA. A solve repeated from the same inputs therefore gives the same bits, with one
iteration per launch and with 64, and so does one whose pivots end below the threshold of 64 eps of the
largest diagonal entry (fewer unknowns than the Krylov blocks span: the breakdown falls in the Xi or zeta step)."""
import numpy as np
import pytest

import workloads as wl

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mb():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2608_07327_gb300 as mb
    mb.lib()
    return mb


def fits(n, nnz, kp=8):
    """The FP64 FMAs of one iteration, which decide about the one-cluster loop."""
    return nnz * kp + n * kp * (2 * (kp // 2 + 1) + 5 * kp + 1) <= 1400000


@pytest.mark.parametrize("name,factory,s,precond", [
    ("poisson55_s8", lambda: wl.poisson2d(55), 8, 0),
    ("poisson50_s5_jacobi", lambda: wl.poisson2d(50), 5, 1),
    ("stencil12_s6", lambda: wl.stencil27(12, 3), 6, 0),
])
def test_launches_of_64_iterations_join(mb, name, factory, s, precond):
    A = factory()
    assert fits(A.n, A.nnz)
    b, U = wl.rhs(A.n, 0), wl.initial_block(A.n, s, 1)
    ends = []
    for mode in (mb.MBPCG_LAUNCH_GRAPH, mb.MBPCG_LAUNCH_EAGER):
        sv = mb.Solver(A, s=s, precond=precond, launch_mode=mode)
        try:
            got = [sv.solve(b, U, tol=1e-15, maxit=m) for m in (1, 63, 64, 65)] + [sv.solve(b, U, tol=1e-8)]
            state, _ = sv.run_iterations(b, U, 40)
        finally:
            sv.close()
        ends.append((got, state))
    for (x, i), (y, j) in zip(ends[0][0], ends[1][0]):
        assert (i["status"], i["iterations"]) == (j["status"], j["iterations"]) and np.array_equal(x, y)
    assert ends[0][0][4][1]["status"] == 0
    for key in ("X0", "Xt", "R", "W", "P", "Sigma"):
        assert np.array_equal(ends[0][1][key], ends[1][1][key]), key


@pytest.mark.parametrize("n,s", [(20, 8), (33, 8), (41, 7), (60, 5)])
def test_pivots_at_the_threshold_decide_alike(mb, n, s):
    """n unknowns are spanned after about n / s iterations: the next Gram matrices are rounding noise."""
    rp = np.arange(n + 1, dtype=np.int32)
    A = wl.CSR(n, rp, rp[:-1].copy(), np.linspace(1.0, 2.0, n))
    b, U = wl.rhs(n, 0), wl.initial_block(n, s, 1)
    sv = mb.Solver(A, s=s)
    try:
        x, info = sv.solve(b, U, tol=1e-30, maxit=200)
        for _ in range(100):
            y, again = sv.solve(b, U, tol=1e-30, maxit=200)
            assert (again["status"], again["iterations"]) == (info["status"], info["iterations"])
            assert np.array_equal(x, y, equal_nan=True)
    finally:
        sv.close()
    assert info["status"] in (mb.MBPCG_NOT_CONVERGED, mb.MBPCG_BREAKDOWN)
