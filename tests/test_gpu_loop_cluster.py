"""Small CSR systems iterate in one thread-block cluster (csrc/loop_cluster.cu): the state against the
oracle's, and what ends a launch or a solve at and around its 64 iterations.

Tolerance of the state: each sum is of FP64 terms in another order than the oracle's, n x 2^-53 of its
largest partial sums at worst (n <= 5,000: 6e-13), times what the k x k steps magnify in the first
iterations of these well-conditioned systems (below 10): 1e-11."""
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


def arrow(n):
    """First row and column full: one CTA has most of the entries, and every CTA reads its first row."""
    D = np.diag(np.linspace(2.0, 3.0, n))
    D[0, 1:] = D[1:, 0] = -1e-3
    D[0, 0] = 3.0
    r, c = np.nonzero(D)
    rp = np.zeros(n + 1, np.int32)
    np.cumsum(np.bincount(r, minlength=n), out=rp[1:])
    return wl.CSR(n, rp, c.astype(np.int32), D[r, c])


# every padded width, fewer rows than CTAs, rows that no CTA count divides, one chunk of a warp more or less,
# rows longer than a batch of 8 entries, scaling; padded columns
CASES = [
    ("diag1_s1", lambda: wl.poisson2d(1), 1, 0, ()),
    ("poisson3_s1", lambda: wl.poisson2d(3), 1, 0, (1, 2)),
    ("poisson4_s2", lambda: wl.poisson2d(4), 2, 0, (1, 2)),
    ("poisson7_s3", lambda: wl.poisson2d(7), 3, 0, (1, 3)),
    ("poisson23_s4", lambda: wl.poisson2d(23), 4, 0, (1, 3)),
    ("poisson32_s1", lambda: wl.poisson2d(32), 1, 0, (1, 4)),
    ("poisson70_s4", lambda: wl.poisson2d(70), 4, 0, (1, 3)),
    ("diffusion13_s2_jacobi", lambda: wl.diffusion3d(13, 1), 2, 1, (1, 3)),
    ("diffusion11_s8_jacobi", lambda: wl.diffusion3d(11, 2), 8, 1, (1, 3)),
    ("diffusion12_s5_jacobi", lambda: wl.diffusion3d(12, 3), 5, 1, (1, 3)),
    ("stencil11_s7", lambda: wl.stencil27(11, 4), 7, 0, (1, 3)),
    ("stencil10_s4", lambda: wl.stencil27(10, 5), 4, 0, (1, 3)),
    ("arrow700_s6", lambda: arrow(700), 6, 0, (1, 2)),
]


@pytest.mark.parametrize("name,factory,s,precond,iters", CASES, ids=[c[0] for c in CASES])
def test_state_and_solution_match_oracle(mb, orc, name, factory, s, precond, iters):
    A = factory()
    b, U = wl.rhs(A.n, 0), wl.initial_block(A.n, s, 1)
    sv = mb.Solver(A, s=s, precond=precond)
    try:
        for m in iters:
            got, st = sv.run_iterations(b, U, m)
            ref, st_o = orc.mbpcg_state(A, b, U, m, precond=precond)
            assert st == st_o
            for key in ("X0", "Xt", "R", "W", "P", "Sigma"):
                scale = np.abs(ref[key]).max()
                assert np.abs(got[key] - ref[key]).max() <= 1e-11 * scale, (key, m)
        x, info = sv.solve(b, U, tol=1e-8)
        x2, info2 = sv.solve(b, U, tol=1e-8)
    finally:
        sv.close()
    assert info["status"] == 0 and info["iterations"] == info2["iterations"] and np.array_equal(x, x2)
    assert np.linalg.norm(b - A.to_scipy() @ x) <= 1e-8 * np.linalg.norm(b)


@pytest.mark.parametrize("s,precond", [(1, 0), (3, 0), (4, 1), (8, 0)])
def test_launches_of_64_iterations_join(mb, s, precond):
    """One launch per iteration (eager) and per 64 (graph) give the same bits, whatever ends the solve:
    the iteration cap before, at and after a launch's end, or the tolerance."""
    A = wl.poisson2d(60)
    b, U = wl.rhs(A.n, 0), wl.initial_block(A.n, s, 1)
    ends = []
    for mode in (mb.MBPCG_LAUNCH_GRAPH, mb.MBPCG_LAUNCH_EAGER):
        sv = mb.Solver(A, s=s, precond=precond, launch_mode=mode)
        try:
            got = [sv.solve(b, U, tol=1e-14, maxit=m) for m in (1, 63, 64, 65)] + [sv.solve(b, U, tol=1e-8)]
            state, _ = sv.run_iterations(b, U, 66)
        finally:
            sv.close()
        ends.append((got, state))
    for (x, i), (y, j) in zip(ends[0][0], ends[1][0]):
        assert (i["status"], i["iterations"]) == (j["status"], j["iterations"]) and np.array_equal(x, y)
    assert [i["iterations"] for _, i in ends[0][0][:4]] == [1, 63, 64, 65]
    assert ends[0][0][4][1]["status"] == 0
    for key in ("X0", "Xt", "R", "W", "P", "Sigma"):
        assert np.array_equal(ends[0][1][key], ends[1][1][key]), key
