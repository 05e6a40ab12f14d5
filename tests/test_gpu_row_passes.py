"""The tensor-core row passes of large CSR handles (csrc/rows_mma.cuh): block update, W/P update and Gram
matrices by digit splitting, against the oracle's FP64 state and solutions.

Tolerance of the state: a row product is off by at most a few 2^-54 of (largest value of the row) x
(largest of the matrix column) x the width, a Gram by as much of its column norms, so one iteration adds
less than 64 * 32 * 2^-54 = 1.2e-13 of a block's largest entry times what the k x k steps magnify (the
condition number of the two Grams, below 100 in the first iterations of these systems): 1e-11."""
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


# every padded width above the rule's line (n kp >= 2^17, the product's Gram at 2^19), with ragged last
# tiles of 16 view rows, an odd n at kp = 4 (half a view row) and padded columns
CASES = [
    ("poisson183_s4", lambda: wl.poisson2d(183), 4, 0, 0),
    ("poisson183_s3_implicit", lambda: wl.poisson2d(183), 3, 0, 1),
    ("diffusion26_s8_jacobi", lambda: wl.diffusion3d(26, 1), 8, 1, 0),
    ("diffusion26_s6_jacobi_implicit", lambda: wl.diffusion3d(26, 1), 6, 1, 1),
    ("poisson91_s16", lambda: wl.poisson2d(91), 16, 0, 0),
    ("stencil21_s11_implicit", lambda: wl.stencil27(21, 2), 11, 0, 1),
    ("diffusion33_s16_jacobi", lambda: wl.diffusion3d(33, 3), 16, 1, 0),
    ("poisson65_s23", lambda: wl.poisson2d(65), 23, 0, 0),
    ("diffusion26_s32_jacobi", lambda: wl.diffusion3d(26, 4), 32, 1, 0),
    ("diffusion26_s20_jacobi_implicit", lambda: wl.diffusion3d(26, 4), 20, 1, 1),
]


@pytest.mark.parametrize("name,factory,s,precond,implicit", CASES, ids=[c[0] for c in CASES])
def test_state_and_solution_match_oracle(mb, orc, name, factory, s, precond, implicit):
    A = factory()
    assert A.n * mb.mbpcg_k_padded_width(s) >= 1 << 17
    b = wl.rhs(A.n, 0)
    U = wl.initial_block(A.n, s, 1)
    sv = mb.Solver(A, s=s, precond=precond, residual_mode=implicit)
    try:
        for m in (1, 3):
            got, st = sv.run_iterations(b, U, m)
            ref, st_o = orc.mbpcg_state(A, b, U, m, precond=precond)
            assert st == st_o == 0
            for key in ("X0", "Xt", "R", "W", "P", "Sigma"):
                scale = np.abs(ref[key]).max()
                assert np.abs(got[key] - ref[key]).max() <= 1e-11 * scale, (key, m)
        x, info = sv.solve(b, U, tol=1e-8)
        x2, _ = sv.solve(b, U, tol=1e-8)
    finally:
        sv.close()
    assert info["status"] == 0 and np.array_equal(x, x2)
    assert np.linalg.norm(b - A.to_scipy() @ x) <= 1e-8 * np.linalg.norm(b)


def test_non_finite_right_hand_side_ends_alike(mb):
    """A NaN in b makes every Gram NaN, whichever path forms it (n = 64^2 takes the FP64 passes, 183^2 the
    tensor-core ones): both end in the set-up's Cholesky QR, in the same way."""
    ends = []
    for m in (64, 183):
        A = wl.poisson2d(m)
        b = wl.rhs(A.n, 0)
        b[7] = np.nan
        sv = mb.Solver(A, s=4)
        try:
            x, info = sv.solve(b, None, tol=1e-8)
        finally:
            sv.close()
        ends.append((info["status"], info["iterations"], info["restarts"], info["ls_fallback"], bool(np.isnan(x).any())))
    assert ends[0] == ends[1]
