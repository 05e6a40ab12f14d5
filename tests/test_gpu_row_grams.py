"""The Gram matrices of the tensor-core passes (csrc/rows_mma.cuh, k_gram_mx) over many tiles per warp: sums drained
every 7 tiles, last tiles of some warps only, and scales that grow from tile to tile (rows rising by 10^6 along n).
The matrix is diagonal, so that n can be any number.

Tolerances. Sigma^T Sigma = R^T R: the Cholesky factorisation is off by (s + 1) 2^-53 of the norms of the columns, both
sums by less than 30 x 2^-53 of them (blocked, a few hundred terms in turn at most, with random signs): (s + 61) 2^-53.
T = Xi Sigma, fitted from X~ = P T by normal equations in FP64: 1e-12 (the condition numbers are below 10)."""
import numpy as np
import pytest

import workloads as wl

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

U53 = 2.0 ** -53


@pytest.fixture(scope="module")
def mb():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2608_07327_gb300 as mb
    mb.lib()
    return mb


def rows_of_tiles(s, tiles):
    """n for which the warps of two CTAs per SM have so many tiles of 16 view rows each."""
    warps = 2 * torch.cuda.get_device_properties(0).multi_processor_count * 8
    kp = 1 << (s - 1).bit_length()
    return int(tiles * warps * 16) * max(1, 16 // kp) + 1


@pytest.mark.parametrize("rise", [0.0, 6.0])
@pytest.mark.parametrize("s,tiles", [(16, 1.4), (16, 6.6), (16, 7.0), (11, 7.5), (16, 14.3), (16, 15.6), (4, 8.3),
                                     (3, 15.5), (8, 15.5), (32, 7.7), (20, 15.2)])
def test_set_up_and_product_grams(mb, s, tiles, rise):
    n = rows_of_tiles(s, tiles)
    rng = np.random.default_rng(n)
    diag = rng.uniform(1.0, 2.0, n)
    rp = np.arange(n + 1, dtype=np.int32)
    ramp = 10.0 ** (rise * np.arange(n) / n)
    b = rng.uniform(-1.0, 1.0, n) * ramp
    U = np.asfortranarray(rng.uniform(-1.0, 1.0, (n, s)) * ramp[:, None])
    sv = mb.Solver(wl.CSR(n, rp, rp[:-1].copy(), diag), s=s)
    try:
        z, _ = sv.run_iterations(b, U, 0)
        one, _ = sv.run_iterations(b, U, 1)
    finally:
        sv.close()
    R, P, Sigma = z["R"], z["P"], z["Sigma"]
    norm = np.sqrt((R ** 2).sum(0))
    assert np.abs(Sigma.T @ Sigma - R.T @ R).max() <= (s + 61) * U53 * norm.max() ** 2
    T = np.linalg.solve(P.T @ (diag[:, None] * P), Sigma)
    fitted = np.linalg.solve(P.T @ P, P.T @ one["Xt"])
    assert np.abs(fitted - T).max() <= 1e-12 * np.abs(T).max()
    S1 = one["Sigma"] @ np.linalg.inv(Sigma)  # zeta of the first iteration: V^T V = zeta^T zeta
    V = P - (diag[:, None] * P) @ np.linalg.solve(P.T @ (diag[:, None] * P), np.eye(s))
    assert np.abs(S1.T @ S1 - V.T @ V).max() <= 1e-12 * np.abs(V.T @ V).max()


@pytest.mark.parametrize("s,tiles", [(4, 7.6), (8, 15.3), (16, 15.4), (32, 7.4)])
def test_weighted_gram_of_the_implicit_residual(mb, s, tiles):
    """||D R_h|| after three iterations from V^T D^2 V (implicit) and from R itself (explicit); D^2 from 1 to 10^4."""
    n = rows_of_tiles(s, tiles)
    rng = np.random.default_rng(n)
    rp = np.arange(n + 1, dtype=np.int32)
    A = wl.CSR(n, rp, rp[:-1].copy(), 10.0 ** rng.uniform(0.0, 4.0, n))
    off = np.arange(0, n - 1, 2)  # pairs of coupled unknowns, or Jacobi scaling leaves the identity
    rows = np.concatenate([np.arange(n), off, off + 1])
    cols = np.concatenate([np.arange(n), off + 1, off])
    couple = -rng.uniform(0.1, 0.9, off.size) * np.sqrt(A.val[off] * A.val[off + 1])
    vals = np.concatenate([A.val, couple, couple])
    order = np.lexsort((cols, rows))
    np.cumsum(np.bincount(rows, minlength=n), out=rp[1:])
    A = wl.CSR(n, rp, cols[order].astype(np.int32), vals[order])
    b, U = wl.rhs(n, 0), wl.initial_block(n, s, 1)
    nu = []
    for mode in (0, 1):
        sv = mb.Solver(A, s=s, precond=1, residual_mode=mode)
        try:
            nu.append(sv.solve(b, U, tol=1e-14, maxit=3)[1]["relres_recurrence"])
        finally:
            sv.close()
    assert abs(nu[0] - nu[1]) <= 1e-12 * nu[0]
