"""The m x m steps of the dense phase at the sizes where their kernels change:
one warp, ragged blocks of eight, the largest width; layout moves on both
sides of the small-block rule, reordered and not.

Rayleigh-Ritz on a block whose Ritz values come in exact multiplicities (three
equal grid sides) and on one with well separated values; tolerances are the
backward errors of an m-column FP64 product, n u with u = 2^-53 and ||A||_1.
"""
import numpy as np
import pytest

from gpu_util import colmajor_dev, from_colmajor
from workloads import graphs as G

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m", [1, 2, 7, 33, 80, 127, 128])
@pytest.mark.parametrize("kind", ["clusters", "random"])
def test_rayleigh_ritz_is_a_decomposition(lib, m, kind):
    import torch
    lap = G.grid3d(11, 11, 11, 0.1)
    A, n = lap.scipy(), lap.n
    rng = np.random.default_rng(m)
    if kind == "random":
        q0 = np.linalg.qr(rng.standard_normal((n, m)))[0]
    else:  # eigenvectors of the grid, rotated among themselves
        import scipy.linalg as sl
        v = sl.eigh(A.toarray(), subset_by_index=[0, m - 1])[1]
        q0 = v @ np.linalg.qr(rng.standard_normal((m, m)))[0]
    h = lib.rafeast_create(lap.row_ptr, lap.col_idx, lap.values, lap.shift)
    try:
        Q = colmajor_dev(q0)
        theta, _ = lib.rafeast_rayleigh_ritz(h, m, Q)
        q = from_colmajor(Q)
        tol = n * 2.0 ** -53 * 12.1
        assert np.all(np.diff(theta) >= 0)
        assert np.abs(q.T @ q - np.eye(m)).max() <= tol
        assert np.abs(q.T @ (A @ q) - np.diag(theta)).max() <= tol
        assert np.linalg.norm(q - q0 @ (q0.T @ q)) <= tol * m
        R = lib.rafeast_orthonormalize(h, m, colmajor_dev(q0 * np.logspace(0, -3, m)), want_r=True)
        assert np.allclose(np.abs(np.diag(R)), np.logspace(0, -3, m), rtol=tol)
    finally:
        lib.rafeast_destroy(h)


@pytest.mark.parametrize("n,k", [(31, 3), (33, 130), (8191, 64), (8193, 65), (20011, 27)])
@pytest.mark.parametrize("flag", [1, 2])  # the caller's row order, a reordering
def test_layout_moves_keep_every_entry(lib, n, k, flag):
    """A x for integer-valued x is exact in FP64, so the product shows that each
    entry went to its place and came back."""
    import torch
    lap = G.cycle(n, 1.0) if hasattr(G, "cycle") else G.grid2d(n, 1, 1.0)
    x = np.arange(n * k, dtype=np.float64).reshape(n, k) % 1021
    h = lib.rafeast_create(lap.row_ptr, lap.col_idx, lap.values, lap.shift, flags=flag)
    try:
        X = colmajor_dev(x)
        Y = torch.full_like(X, -1.0)
        lib.rafeast_spmm(h, k, 1.0, 0.0, X, Y)
        assert np.array_equal(from_colmajor(Y), lap.scipy() @ x)
    finally:
        lib.rafeast_destroy(h)


@pytest.mark.parametrize("m", [1, 15, 16, 17, 32, 33, 48, 49, 64, 65, 96, 127, 128])
def test_block_product_widths(lib, m):
    """A X over every chunk count and column-block count of the product's
    instances, with a row longer than one group's index load; a row of d entries
    and the shift is a chain of d + 2 roundings."""
    import torch
    lap = G.knn3d(333, 10, seed=4, shift=0.7)
    A = lap.scipy().tocsr()
    x = np.random.default_rng(m).standard_normal((lap.n, m))
    h = lib.rafeast_create(lap.row_ptr, lap.col_idx, lap.values, lap.shift)
    try:
        X = colmajor_dev(x)
        Y = torch.full_like(X, 7.0)
        lib.rafeast_spmm(h, m, 1.0, 0.0, X, Y, lib.RAFEAST_FP64)
        d = np.diff(A.indptr)[:, None] + 2
        assert np.all(np.abs(from_colmajor(Y) - A @ x) <= 2 * d * 2.0 ** -53 * (abs(A) @ np.abs(x)))
    finally:
        lib.rafeast_destroy(h)


@pytest.mark.parametrize("n", [140, 601, 9800])
@pytest.mark.parametrize("m", [1, 15, 16, 17, 33, 64, 65, 127, 128])
def test_preconditioned_orthonormalisation_widths(lib, m, n):
    """The warmstart's Cholesky-QR passes (the first of each with a float Gram)
    at the edges of the Gram's 16-column blocks, with row ranges shorter than a
    stage, ragged and of several stages: an orthonormal basis whose Ritz values
    are those of A on it. Backward errors as above, n u ||A||_1, and eight roundings
    for each of up to 128 columns."""
    lap = G.knn3d(n, 10, seed=6, shift=0.1)
    A = lap.scipy()
    h = lib.rafeast_create(lap.row_ptr, lap.col_idx, lap.values, lap.shift)
    try:
        lib.rafeast_warmstart(h, 0.05, 1.0, m, 0, 1, 3)
        Q = np.zeros((m, n))
        theta = lib.rafeast_get_subspace(h, Q, m)
        q, tol = Q.T, (n + 8 * 128) * 2.0 ** -53 * abs(A).sum(0).max()
        assert np.abs(q.T @ q - np.eye(m)).max() <= tol
        assert np.abs(q.T @ (A @ q) - np.diag(theta)).max() <= tol
    finally:
        lib.rafeast_destroy(h)


@pytest.mark.parametrize("gap", [0.0, 1.0, 32.0])
@pytest.mark.parametrize("m", [3, 16, 80])
def test_close_pair_far_below_the_others_is_resolved(lib, m, gap):
    """Two eigenvalues near 2^-30 beside ones of order 1, joined by an entry b of
    a few units of rounding of the large ones, gap b apart: delta + gap b / 2 +-
    b sqrt(1 + gap^2 / 4). The block is unit vectors, so every product up to the
    eigensolver is exact, the float stage finds nothing to rotate (b is below its
    threshold) and one rotation of the pair remains: eight roundings of delta are
    2^-50 delta, 2^-80, against b of about 2^-50."""
    n, delta = 200, 2.0 ** -30
    d = np.full(n, 3.0)
    d[:m] = 1.0 + np.arange(m)[::-1] / m
    rms = np.sqrt((d[2:m] ** 2).sum() / m)
    b = 2.0 ** -52 * (2.0 if m == 3 else 6.0) * 2.0 ** np.floor(np.log2(rms))
    d[0], d[1] = delta, delta + gap * b
    rows = [[(i, d[i])] for i in range(n)]
    rows[0].append((1, b))
    rows[1].insert(0, (0, b))
    rp = np.cumsum([0] + [len(r) for r in rows]).astype(np.int32)
    ci = np.array([c for r in rows for c, _ in r], dtype=np.int32)
    v = np.array([x for r in rows for _, x in r])
    q0 = np.zeros((n, m))
    q0[np.arange(m), np.arange(m)] = 1.0
    h = lib.rafeast_create(rp, ci, v, 0.0)
    try:
        Q = colmajor_dev(q0)
        theta, _ = lib.rafeast_rayleigh_ritz(h, m, Q)
        q = from_colmajor(Q)
    finally:
        lib.rafeast_destroy(h)
    root = b * np.sqrt(1.0 + gap * gap / 4.0)
    exp = delta + gap * b / 2.0 + np.array([-root, root])
    assert np.max(np.abs(theta[:2] - exp)) <= 2.0 ** -50 * delta
    # (b, theta - delta) up to scale is an eigenvector: the angle is the same to
    # 2^-50 delta / b < 2^-28
    ang = np.arctan2(np.abs(q[1, :2]), np.abs(q[0, :2]))
    assert np.max(np.abs(ang - np.arctan2(np.abs(exp - delta), b))) <= 2.0 ** -28


@pytest.mark.parametrize("k", [1, 2, 13, 14, 15, 16])
@pytest.mark.parametrize("flag", [1, 2])
def test_narrow_layout_moves_keep_every_entry(lib, k, flag):
    """As test_layout_moves_keep_every_entry, on both sides of the line between
    narrow blocks and others where there are more than 2^19 elements (524,309 is
    odd: ragged last rows)."""
    import torch
    n = 524309 if k < 8 else 40009
    lap = G.cycle(n, 1.0) if hasattr(G, "cycle") else G.grid2d(n, 1, 1.0)
    x = np.arange(n * k, dtype=np.float64).reshape(n, k) % 1021
    h = lib.rafeast_create(lap.row_ptr, lap.col_idx, lap.values, lap.shift, flags=flag)
    try:
        X = colmajor_dev(x)
        Y = torch.full_like(X, -1.0)
        lib.rafeast_spmm(h, k, 1.0, 0.0, X, Y)
        assert np.array_equal(from_colmajor(Y), lap.scipy() @ x)
    finally:
        lib.rafeast_destroy(h)


@pytest.mark.parametrize("m", [3, 8, 15, 16, 17])
@pytest.mark.parametrize("kind", ["clusters", "random"])
def test_rayleigh_ritz_where_the_refinement_changes_kernel(lib, m, kind):
    """One CTA refines up to 16 columns, products over all SMs more."""
    test_rayleigh_ritz_is_a_decomposition(lib, m, kind)


def test_triangular_block_keeps_its_factor(lib):
    """Columns r e_0 and k e_0 + e_1 with whole r, k: the Gram matrix and both
    Cholesky columns are exact when the pivot column is divided by r, and r (1/r)
    is 1 for these r, so R comes back without an error. A product with a rounded
    1/r misses k by one rounding."""
    pairs = [(75, 15), (77, 15), (93, 29), (99, 29), (150, 15), (154, 15), (186, 29), (191, 15),
             (198, 29), (211, 29), (221, 22), (221, 29), (227, 15), (227, 22), (245, 29), (300, 15),
             (308, 15), (372, 29), (382, 15), (391, 29), (393, 15), (396, 29)]
    n = 64
    rp, ci = np.arange(n + 1, dtype=np.int32), np.arange(n, dtype=np.int32)
    h = lib.rafeast_create(rp, ci, np.ones(n), 0.0)
    try:
        for r, k in pairs:
            x = np.zeros((n, 2))
            x[0, 0], x[0, 1], x[1, 1] = r, k, 1.0
            R = lib.rafeast_orthonormalize(h, 2, colmajor_dev(x), want_r=True)
            assert np.array_equal(R, [[r, k], [0.0, 1.0]]), (r, k, R)
    finally:
        lib.rafeast_destroy(h)
