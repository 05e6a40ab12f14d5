"""CSR CG with its three sums in the product (short rows, or a small system) and apart (long rows of a large
system), against the oracle's CG after 10 iterations.

A dot product of n <= 150,000 terms is off by at most n 2^-53 = 1.7e-11 of its absolute terms on either side, and
10 iterations of these well-conditioned systems add these up: 1e-9 of the solution."""
import numpy as np
import pytest

import workloads as wl

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name,factory,precond", [
    ("stencil49_sums_in_product", lambda: wl.stencil27(49, 1), 0),
    ("stencil52_sums_apart", lambda: wl.stencil27(52, 1), 0),
    ("stencil52_jacobi_sums_apart", lambda: wl.stencil27(52, 1), 1),
    ("diffusion52_jacobi_sums_in_product", lambda: wl.diffusion3d(52, 1), 1),
])
def test_cg_after_ten_iterations(orc, name, factory, precond):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2608_07327_gb300 as mb
    A = factory()
    b = wl.rhs(A.n, 0)
    sv = mb.Solver(A, s=1, precond=precond, algo=1)
    try:
        x, info = sv.solve(b, None, tol=1e-14, maxit=10)
        y, _ = sv.solve(b, None, tol=1e-14, maxit=10)
    finally:
        sv.close()
    xo, io = orc.cg_cgear(A, b, precond=precond, tol=1e-14, maxit=10)
    assert info["iterations"] == io["iterations"] == 10 and np.array_equal(x, y)
    assert np.linalg.norm(x - xo) <= 1e-9 * np.linalg.norm(xo)


def test_two_columns_with_long_rows(orc):
    """The product's Gram by tiles (more than 2^19 rows of more than 16 entries, s = 2): the state after one
    iteration. Sums of n <= 532,000 terms, off by n 2^-53 = 6e-11 at worst on either side: 1e-9."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2608_07327_gb300 as mb
    A = wl.stencil27(81, 2)
    assert A.n > 1 << 19 and A.nnz > 16 * A.n
    b, U = wl.rhs(A.n, 0), wl.initial_block(A.n, 2, 1)
    sv = mb.Solver(A, s=2)
    try:
        got, st = sv.run_iterations(b, U, 1)
    finally:
        sv.close()
    ref, st_o = orc.mbpcg_state(A, b, U, 1)
    assert st == st_o == 0
    for key in ("X0", "Xt", "R", "W", "P", "Sigma"):
        assert np.abs(got[key] - ref[key]).max() <= 1e-9 * np.abs(ref[key]).max(), key
