"""The row products of the tensor-core passes (csrc/rows_mma.cuh) keep the precision of FP64 rows: measured on the
state itself, without the k x k steps that made its factors. After one iteration X~ = P T with P = W of the set-up,
and W = R Sigma^-1 after the set-up; the small factor is fitted to all rows in extended precision, and what a
row is off from the fitted product is the row product's own error."""
import numpy as np
import pytest

import workloads as wl

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

LD = np.longdouble
U53 = 2.0 ** -53


@pytest.fixture(scope="module")
def mb():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2608_07327_gb300 as mb
    mb.lib()
    return mb


def product(X, M):
    """X M in extended precision."""
    return sum(X[:, l:l + 1].astype(LD) * M[l:l + 1].astype(LD) for l in range(X.shape[1]))


def solve_ld(G, B):
    """G^-1 B by Gaussian elimination in extended precision (G small, positive definite)."""
    G, B = G.astype(LD).copy(), B.astype(LD).copy()
    k = len(G)
    for j in range(k):
        for i in range(j + 1, k):
            f = G[i, j] / G[j, j]
            G[i, j:] -= f * G[j, j:]
            B[i] -= f * B[j]
    for j in range(k - 1, -1, -1):
        B[j] = (B[j] - (G[j, j + 1:, None] * B[j + 1:]).sum(0)) / G[j, j]
    return B


def fit(X, Y):
    """The M that minimises |X M - Y|, columns of X brought to like size first."""
    c = np.sqrt((X.astype(LD) ** 2).sum(0))
    Xs = X / c

    def gram(Z):
        return np.stack([(Xs[:, l:l + 1] * Z).sum(0) for l in range(X.shape[1])])

    return solve_ld(gram(Xs), gram(Y.astype(LD))) / c[:, None]


def scaled_grid(m, c):
    """D (I + 0.05 L) D with L the five-point Laplacian on m x m and D alternating 1 and c: two unknowns
    per cell in different units."""
    L = wl.poisson2d(m)
    d = np.where(np.arange(L.n) % 2 == 0, 1.0, c)
    rows = np.repeat(np.arange(L.n), np.diff(L.row_ptr))
    val = 0.05 * L.val
    val[rows == L.col_idx] += 1.0
    return wl.CSR(L.n, L.row_ptr, L.col_idx, val * d[rows] * d[L.col_idx])


def states(mb, A, b, U, s, precond, iters):
    sv = mb.Solver(A, s=s, precond=precond)
    try:
        return [sv.run_iterations(b, U, m)[0] for m in iters]
    finally:
        sv.close()


@pytest.mark.parametrize("s", [3, 4])
def test_neighbouring_rows_of_different_size(mb, s):
    """Each entry within s^2 2^-53 of its row's largest value times its column's: what s FMAs of FP64 may be off
    (each by 2^-53 of a partial sum of at most s such terms)."""
    A = scaled_grid(183, 1e6)
    n = A.n
    assert n * 4 >= 1 << 17
    z, one = states(mb, A, wl.rhs(n, 0), wl.initial_block(n, s, 1), s, 0, (0, 1))
    big = np.abs(z["P"]).max(1, keepdims=True)
    assert big.max() > 1e4 * big.min()  # the rows do differ
    P, X = z["P"] / big, one["Xt"] / big
    T = fit(P, X)
    err = np.abs(product(P, T) - X).max(0) / np.abs(T).max(0)
    assert (err <= s * s * U53).all(), err


@pytest.mark.parametrize("name,factory,s,precond", [
    ("stencil26_s8", lambda: wl.stencil27(26, 1), 8, 0),
    ("diffusion26_s16_jacobi", lambda: wl.diffusion3d(26, 2), 16, 1),
    ("poisson92_s23", lambda: wl.poisson2d(92), 23, 0),
    ("stencil21_s32", lambda: wl.stencil27(21, 3), 32, 0),
    ("diffusion21_s32_jacobi", lambda: wl.diffusion3d(21, 4), 32, 1),
])
def test_products_are_off_by_little_more_than_their_rounding(mb, name, factory, s, precond):
    """Root mean square of the errors of W = R Sigma^-1 and X~ = P T against that of the values. Rounding the result
    to FP64 gives 0.43 x 2^-53 and splitting into digits adds a tenth of that; the sums of an FP64 pass are off by
    more the more columns they have. The bound is 2^-53."""
    A = factory()
    assert A.n * mb.mbpcg_k_padded_width(s) >= 1 << 17
    z, one = states(mb, A, wl.rhs(A.n, 0), wl.initial_block(A.n, s, 1), s, precond, (0, 1))
    for X, Y in ((z["R"], z["W"]), (z["W"], one["Xt"])):
        E = product(X, fit(X, Y)) - Y
        assert np.sqrt((E ** 2).sum() / (Y.astype(LD) ** 2).sum()) <= U53


@pytest.mark.parametrize("s", [16, 25, 32])
def test_product_gram_of_rows_in_different_units(mb, s):
    """P is small where A P is large: P^T (A P) = G has terms of one size in rows whose factors are 10^6 apart. T = Xi
    Sigma, fitted from X~ = P T, against G^-1 Sigma in extended precision. A sum of FP64 terms by at most 30 rows in
    turn is off by 30 x 2^-53, the k x k steps add at most 8 s x 2^-53, and G^-1 magnifies both by its condition."""
    scipy_linalg = pytest.importorskip("scipy.sparse.linalg")
    A = scaled_grid(183, 1e6)
    S = A.to_scipy().tocsc()
    n, d = A.n, np.sqrt(S.diagonal())
    assert n * mb.mbpcg_k_padded_width(s) >= 1 << 19
    rows = wl.initial_block(n, s + 1, 1) / (d / d.min())[:, None]
    b = rows[:, s].copy()
    U = np.asfortranarray(scipy_linalg.splu(S).solve(b[:, None] - rows[:, :s]))
    z, one = states(mb, A, b, U, s, 0, (0, 1))
    P = z["W"].astype(LD)
    Q = np.zeros_like(P)
    for i in range(int(np.diff(A.row_ptr).max())):  # A P in extended precision, entry i of every row
        at = A.row_ptr[:-1] + i
        ok = at < A.row_ptr[1:]
        Q[ok] += A.val[at[ok], None].astype(LD) * P[A.col_idx[at[ok]]]
    assert np.abs(Q).max(1).max() > 1e5 * np.abs(P).max()  # the factors do differ
    G = np.stack([(P[:, l:l + 1] * Q).sum(0) for l in range(s)])
    ref = solve_ld(G, z["Sigma"])
    T = fit(z["W"], one["Xt"])
    cond = np.linalg.cond(G.astype(np.float64))
    assert cond < 4
    assert np.abs(T - ref).max() <= (30 + 8 * s) * U53 * cond * np.abs(ref).max()


@pytest.mark.parametrize("s", [4, 8, 13, 32])
def test_columns_of_different_size(mb, s):
    """First residuals from 10^-5 to 1 of b (U_j solves A U_j = b - r_j; the last one is stretched so that the
    set-up's common factor of U, sqrt(s) |b| / |A U|, is 1): W = R Sigma^-1 column by column within 2^-53 in the root
    mean square (an FP64 product with a graded Sigma^-1 is a rounding and little more)."""
    scipy_linalg = pytest.importorskip("scipy.sparse.linalg")
    A = wl.poisson2d(183)
    r = wl.initial_block(A.n, s, 1) * 10.0 ** (np.arange(s) * 5.0 / (s - 1) - 5.0)
    b = wl.rhs(A.n, 0)
    AU = b[:, None] - r
    AU[:, -1] *= np.sqrt((s * (b ** 2).sum() - (AU[:, :-1] ** 2).sum()) / (AU[:, -1] ** 2).sum())
    U = np.asfortranarray(scipy_linalg.splu(A.to_scipy().tocsc()).solve(AU))
    (z,) = states(mb, A, b, U, s, 0, (0,))
    size = np.sqrt((z["R"] ** 2).sum(0))
    assert size.max() > 1e4 * size.min()  # the columns do differ
    W = z["W"].astype(LD)
    E = product(z["R"], fit(z["R"], W)) - W
    assert (np.sqrt((E ** 2).sum(0) / (W ** 2).sum(0)) <= U53).all()


@pytest.mark.parametrize("s", [4, 11, 32])
def test_smooth_column_beside_rough_ones(mb, s):
    """The first residual is smooth, the others are not: the first column of A P is 10^3 to 10^4 below the others, and
    Xi makes up for it. R = R_0 - (A P) T column by column: every one of s FMAs rounds to 2^-53 of a partial sum, which
    is at most |R_0| + sum_l |(A P)_l| |T_lj|."""
    A = wl.poisson2d(183)
    n = A.n
    x = np.sin(np.pi * np.arange(1, 184) / 184)
    smooth = np.outer(x, x).ravel()
    b = smooth + 1e-5 * wl.rhs(n, 0)
    U = wl.initial_block(n, s, 1)
    U[:, 0] = -100.0 * smooth
    z, one = states(mb, A, b, U, s, 0, (0, 1))
    P = torch.zeros((n, mb.mbpcg_k_padded_width(s)), dtype=torch.float64, device="cuda")
    P[:, :s] = torch.as_tensor(z["P"], device="cuda")
    sv = mb.Solver(A, s=s)
    try:
        Q = sv.apply(P)[:, :s].cpu().numpy()  # the loop's A P, bit for bit
    finally:
        sv.close()
    size = np.sqrt((Q ** 2).sum(0))
    assert size.max() > 1e3 * size[0]
    D = z["R"].astype(LD) - one["R"]
    T = fit(Q, D)
    E = product(Q, T) - D
    bound = np.sqrt((z["R"] ** 2).sum(0)) + (size[:, None] * np.abs(T)).sum(0)
    err = np.sqrt((E ** 2).sum(0)) / bound
    assert (err <= s * U53).all(), err / U53


@pytest.mark.parametrize("s", [4, 8, 16, 32])
@pytest.mark.parametrize("value", [np.nan, -np.inf])
def test_non_finite_initial_block_breaks_down_at_the_set_up(mb, s, value):
    """One value of U that is not finite makes the first residual's Gram matrix NaN: its Cholesky factor has no
    positive pivot, and no iteration is made."""
    A = wl.poisson2d(183)
    b, U = wl.rhs(A.n, 0), wl.initial_block(A.n, s, 1)
    U[20000, s - 1] = value
    sv = mb.Solver(A, s=s)
    try:
        _, info = sv.solve(b, U, tol=1e-8)
    finally:
        sv.close()
    assert (info["status"], info["iterations"]) == (mb.MBPCG_BREAKDOWN, 0)


@pytest.mark.parametrize("s,precond", [(4, 0), (8, 0), (16, 0), (11, 1), (32, 0)])
@pytest.mark.parametrize("power", [-400, 400])
def test_a_power_of_two_changes_no_bit(mb, s, precond, power):
    """2^400 A and 2^-400 A: the scales follow, every digit stays. X0 and X~ are 2^-power of those of A, R, W, P and
    Sigma the same (unscaled; Jacobi scaling takes D = 2^(power / 2) out of X and R besides)."""
    A = wl.diffusion3d(33, 6) if s > 4 else wl.diffusion3d(41, 6)
    n = A.n
    b, U = wl.rhs(n, 0), wl.initial_block(n, s, 1)
    (one,) = states(mb, A, b, U, s, precond, (2,))
    B = wl.CSR(n, A.row_ptr, A.col_idx, A.val * 2.0 ** power)
    (two,) = states(mb, B, b, U, s, precond, (2,))
    half = 2.0 ** (-power // 2)
    factor = {"X0": 2.0 ** -power, "Xt": 2.0 ** -power, "R": 1.0, "W": 1.0, "P": 1.0, "Sigma": 1.0}
    if precond:
        factor = {"X0": half, "Xt": half, "R": half, "W": 1.0, "P": 1.0, "Sigma": half}
    for key, f in factor.items():
        assert np.array_equal(two[key], one[key] * f), key
