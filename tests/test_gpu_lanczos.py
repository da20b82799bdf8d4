"""Real Lanczos form of the multi-shift filter (the default route) against the
oracle's conjugate orthogonal CG after a fixed number of steps.

The ring holds every step here, so one pass over it ends the filter (rings that
are folded: test_gpu_ring.py). The step counts lie at the edges of 32 steps, the
slots of a slab and the rows of the collapse's tiles; the widths leave ragged
16-byte chunks of columns and ragged column blocks; the node counts fill one to
twelve lanes of the warp that has a column's nodes. solve_tol = 0: every system runs to the cap.

Tolerance (backward errors): a step rounds each value a few times (2^2), which
is an error of the matrix of at most 2^2 eps ||A|| per step; k <= 70 steps make
2^2 k < 2^9 of it. It changes x_j = (z_j - A)^-1 q by at most
2^9 eps ||A|| / Im(z_j) times ||x_j|| <= ||q|| / Im(z_j), so the error of a
column of unit norm is at most
2^9 eps ||A|| sum_j |w_j| / Im(z_j)^2. On a grid no Ritz value converges within
these steps, so the recurrence itself amplifies nothing.
"""
import numpy as np
import pytest

from gpu_util import colmajor_dev, from_colmajor
from oracle import feast as OF
from oracle import quadrature as OQ
from workloads import graphs as G

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("values_free", [0, 1])
@pytest.mark.parametrize("steps", [1, 31, 32, 33, 70])
@pytest.mark.parametrize("m0,nc", [(1, 1), (5, 2), (46, 3), (80, 4), (17, 8), (97, 12)])
def test_fixed_steps_match_oracle(lib, m0, nc, steps, values_free):
    import torch
    lap = G.grid2d(37, 41, shift=0.3)
    A, n, (lo, hi) = lap.scipy(), lap.n, (0.31, 0.6)
    q0 = OF.random_start(n, m0, 1)
    z, w = OQ.nodes(lo, hi, nc, 1.0)
    exp, _ = OF.filter_apply(A, q0, z, w, 0.0, steps, "direct")
    bound = 2.0 ** 9 * OF.one_norm(A) * np.sum(np.abs(w) / z.imag ** 2)
    h = lib.rafeast_create(lap.row_ptr, lap.col_idx, lap.values, lap.shift)
    try:
        lib.rafeast_set_option(h, lib.RAFEAST_OPT_VALUES_FREE, values_free)
        for prec, tiled, eps in ((lib.RAFEAST_FP64, 1, 2.0 ** -52), (lib.RAFEAST_MIXED, 1, 2.0 ** -23),
                                 (lib.RAFEAST_MIXED, 2, 2.0 ** -23)):
            lib.rafeast_set_option(h, lib.RAFEAST_OPT_TILED, tiled)
            prm = lib.make_params(lo, hi, m0, nc, 1.0, 0.0, 1e-10, 1, steps, prec,
                                  lib.RAFEAST_FORM_DIRECT)
            Q = colmajor_dev(q0)
            Qt = torch.zeros_like(Q)
            info = lib.rafeast_filter(h, prm, Q, None, Qt)
            assert info.cocg_min_last == info.cocg_max_last == steps
            err = np.linalg.norm(from_colmajor(Qt) - exp, axis=0)
            assert np.max(err) <= bound * eps, (prec, tiled, float(np.max(err)))
    finally:
        lib.rafeast_destroy(h)


def test_zero_column_and_nan_input(lib):
    """A zero column stops at step 0 with a zero result; a NaN column is
    reported as a breakdown, as by the COCG kernels."""
    import torch
    lap = G.grid2d(20, 23, shift=0.3)
    q0 = OF.random_start(lap.n, 6, 2)
    q0[:, 2] = 0.0
    h = lib.rafeast_create(lap.row_ptr, lap.col_idx, lap.values, lap.shift)
    try:
        for prec in (lib.RAFEAST_FP64, lib.RAFEAST_MIXED):
            prm = lib.make_params(0.31, 0.6, 6, 4, 1.0, 1e-3, 1e-10, 1, 200, prec, lib.RAFEAST_FORM_DIRECT)
            Q = colmajor_dev(q0)
            Qt = torch.full_like(Q, 7.0)
            lib.rafeast_filter(h, prm, Q, None, Qt)
            got = from_colmajor(Qt)
            assert np.all(got[:, 2] == 0.0) and np.all(np.isfinite(got))
            Q[4, 5] = float("nan")
            with pytest.raises(lib.RafeastError) as ei:
                lib.rafeast_filter(h, prm, Q, None, Qt)
            assert ei.value.code == lib.RAFEAST_ERR_COCG_BREAKDOWN
    finally:
        lib.rafeast_destroy(h)


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
def test_batched_filter_matches_one_at_a_time(lib, prec):
    """Two outer iterations of a batch of uneven grids (one row block to many;
    problems that stop at different steps) against rafeast_solve on the same
    start: the grouped launches change only the order of the sums."""
    shapes, m0s = [(5, 7), (20, 23), (37, 41), (90, 101)], [3, 8, 17, 30]
    p = lib.RAFEAST_FP64 if prec == "fp64" else lib.RAFEAST_MIXED
    laps = [G.grid2d(a, b, shift=0.1 * (t + 1)) for t, (a, b) in enumerate(shapes)]
    prms = [lib.make_params(0.05, 0.1 * (t + 1) + 0.3, m, 3, 0.5, 1e-3, 0.0, 2, 40 + 13 * t, p,
                            lib.RAFEAST_FORM_CORRECTION, lib.RAFEAST_START_RANDOM, 5)
            for t, m in enumerate(m0s)]
    hs = [lib.rafeast_create(x.row_ptr, x.col_idx, x.values, x.shift) for x in laps]
    h1 = [lib.rafeast_create(x.row_ptr, x.col_idx, x.values, x.shift) for x in laps]
    try:
        ev = [np.zeros(m) for m in m0s]
        _, mf, _ = lib.rafeast_solve_batched(hs, prms, ev)
        for t, m in enumerate(m0s):
            e1 = np.zeros(m)
            _, mf1, _ = lib.rafeast_solve(h1[t], prms[t], e1)
            assert mf1 == mf[t]
            # Ritz values after two filters: errors enter squared; 2^9 units of
            # the working precision of the filter, relative to ||A||_1 < 8.5
            eps = 2.0 ** -52 if prec == "fp64" else 2.0 ** -23
            assert np.max(np.abs(np.sort(ev[t]) - np.sort(e1))) <= 2.0 ** 9 * eps * 8.5
    finally:
        for h in hs + h1:
            lib.rafeast_destroy(h)


def test_columns_of_extreme_norm(lib):
    """The filter is linear: FP64 columns times 2^-332 and 2^332 (squared norms
    within the double range, their products not) give the same results times
    that. Scaling by powers of two rounds nothing, so the two results differ by
    the order of the sums alone: 2^9 eps of test_fixed_steps_match_oracle's
    bound each."""
    import torch
    lap = G.grid2d(37, 41, shift=0.3)
    q0 = OF.random_start(lap.n, 6, 3)
    scale = np.array([1.0, 2.0 ** -332, 2.0 ** 332])
    z, w = OQ.nodes(0.31, 0.6, 2, 1.0)
    bound = 2.0 ** 10 * 2.0 ** -52 * OF.one_norm(lap.scipy()) * np.sum(np.abs(w) / z.imag ** 2)
    h = lib.rafeast_create(lap.row_ptr, lap.col_idx, lap.values, lap.shift)
    try:
        out = []
        for x in scale:
            prm = lib.make_params(0.31, 0.6, 6, 2, 1.0, 0.0, 1e-10, 1, 40, lib.RAFEAST_FP64,
                                  lib.RAFEAST_FORM_DIRECT)
            Q = colmajor_dev(q0 * x)
            Qt = torch.zeros_like(Q)
            lib.rafeast_filter(h, prm, Q, None, Qt)
            out.append(from_colmajor(Qt) / x)
        for y in out[1:]:
            assert np.max(np.linalg.norm(y - out[0], axis=0)) <= bound
    finally:
        lib.rafeast_destroy(h)


def _dense_graph(kind):
    rng = np.random.default_rng(5)
    if kind == "knn":
        return G.knn3d(601, 10, seed=2, shift=0.2)
    if kind == "rgg":
        return G.rgg2d(1500, seed=3, shift=0.2)
    if kind == "complete":
        i, j = np.triu_indices(97, 1)
        return G._from_edges(97, i, j, 0.2, "complete")
    # one vertex joined to all of a circulant graph of eight neighbours a vertex
    n, t = 700, np.arange(1, 700)
    i = np.concatenate([np.zeros(699, int)] + [t] * 4)
    j = np.concatenate([t] + [1 + (t - 1 + d) % 699 for d in (1, 2, 3, 5)])
    return G._from_edges(n, i, j, 0.2, "hub")


@pytest.mark.parametrize("m0,nc", [(6, 2), (7, 8), (46, 3), (69, 4)])
@pytest.mark.parametrize("kind", ["knn", "rgg", "complete", "hub"])
def test_fixed_point_sums_against_dense(lib, kind, m0, nc):
    """FP64 filter of unit-weight graphs with eight or more neighbours a row
    (neighbour sums in 64-bit integers) against a dense solve: random columns,
    one unit vector (the largest entry a column can have), a constant one (no
    residual after the first step), columns of norm 1e-100 and 1e100, one of
    entries from 1e-300 to 1.

    Tolerance per unit of ||q||: the stopping rule leaves a residual of 1e-12
    and the recurrence at most 2^2 eps ||A|| ||x|| per step, so the error of
    x_j is at most (1e-12 + steps 2^2 eps ||A|| / Im(z_j)) / Im(z_j)."""
    import torch
    lap = _dense_graph(kind)
    A, n, (lo, hi) = lap.scipy().toarray(), lap.n, (0.1, 4.1)
    q = OF.random_start(n, m0, 1)
    q[:, 0] = 0.0
    q[n // 3, 0] = 1.0
    q[:, 1] = n ** -0.5
    q[:, 2] *= 1e-100
    q[:, 3] *= 1e100
    q[:, 4] = 10.0 ** np.linspace(-300, 0, n)
    z, w = OQ.nodes(lo, hi, nc, 1.0)
    exp = sum((wj * np.linalg.solve(zj * np.eye(n) - A, q)).real for zj, wj in zip(z, w))
    h = lib.rafeast_create(lap.row_ptr, lap.col_idx, lap.values, lap.shift)
    try:
        prm = lib.make_params(lo, hi, m0, nc, 1.0, 1e-12, 1e-10, 1, 2000, lib.RAFEAST_FP64,
                              lib.RAFEAST_FORM_DIRECT)
        Q = colmajor_dev(q)
        Qt = torch.zeros_like(Q)
        info = lib.rafeast_filter(h, prm, Q, None, Qt)
        assert info.cocg_max_last < 2000
        got = from_colmajor(Qt)
    finally:
        lib.rafeast_destroy(h)
    norm = np.linalg.norm(q, axis=0)
    per_step = 4.0 * 2.0 ** -52 * np.abs(A).sum(0).max() * (info.cocg_max_last + 1)
    tol = np.sum(np.abs(w) * (1e-12 + per_step / z.imag) / z.imag)
    assert np.max(np.linalg.norm(got - exp, axis=0) / norm) <= tol


@pytest.mark.parametrize("kind", ["knn", "rgg"])
def test_fixed_point_sums_to_the_end_of_the_range(lib, kind):
    """Columns whose squared norms come near the end of the double range, where
    the bound on the fixed-point sums leaves it before the sums of the
    recurrence do: a filter is refused as a breakdown or is right, and it is
    right up to 2^490 (the greatest degrees are 19 and 70, so ||L||^2 <= 2^15 and
    w^T w stays in the range up to about 2^504). Tolerance: that of
    test_fixed_point_sums_against_dense (the powers of two round nothing)."""
    import torch
    lap = _dense_graph(kind)
    A, n, (lo, hi), m0, nc = lap.scipy().toarray(), lap.n, (0.1, 4.1), 6, 4
    q = OF.random_start(n, m0, 1)
    z, w = OQ.nodes(lo, hi, nc, 1.0)
    exp = sum((wj * np.linalg.solve(zj * np.eye(n) - A, q)).real for zj, wj in zip(z, w))
    h = lib.rafeast_create(lap.row_ptr, lap.col_idx, lap.values, lap.shift)
    try:
        prm = lib.make_params(lo, hi, m0, nc, 1.0, 1e-12, 1e-10, 1, 2000, lib.RAFEAST_FP64,
                              lib.RAFEAST_FORM_DIRECT)
        for e in [0, 490] + list(range(498, 512)):
            x = 2.0 ** e
            Q = colmajor_dev(q * x)
            Qt = torch.zeros_like(Q)
            try:
                info = lib.rafeast_filter(h, prm, Q, None, Qt)
            except lib.RafeastError as err:
                assert err.code == lib.RAFEAST_ERR_COCG_BREAKDOWN and e > 490
                continue
            err = np.linalg.norm(from_colmajor(Qt) / x - exp, axis=0)
            per_step = 4.0 * 2.0 ** -52 * np.abs(A).sum(0).max() * (info.cocg_max_last + 1)
            assert info.cocg_max_last < 2000
            assert np.max(err) <= np.sum(np.abs(w) * (1e-12 + per_step / z.imag) / z.imag), e
    finally:
        lib.rafeast_destroy(h)


@pytest.mark.parametrize("prec,e", [("fp64", 512), ("fp64", 600), ("mixed", 70), ("mixed", 100)])
@pytest.mark.parametrize("solver,update", [(1, 0), (1, 1), (1, 2), (0, 0)])
def test_columns_whose_squared_norm_overflows_are_refused(lib, solver, update, prec, e):
    """||b||^2 outside the range of the working precision: no residual can be
    compared with it, so no column has converged (an infinite ||r||^2 <= an
    infinite bound would say so at step 0, with a zero result). (fp64 2^512 times
    a norm of 2; float entries of about 2^65 and more square to over 2^128.)"""
    import torch
    lap = G.grid2d(20, 23, shift=0.3)
    q0 = 2.0 * OF.random_start(lap.n, 6, 2)
    h = lib.rafeast_create(lap.row_ptr, lap.col_idx, lap.values, lap.shift)
    try:
        lib.rafeast_set_option(h, lib.RAFEAST_OPT_SOLVER, solver)
        lib.rafeast_set_option(h, lib.RAFEAST_OPT_UPDATE, update)
        prm = lib.make_params(0.31, 0.6, 6, 4, 1.0, 1e-3, 1e-10, 1, 200,
                              lib.RAFEAST_FP64 if prec == "fp64" else lib.RAFEAST_MIXED,
                              lib.RAFEAST_FORM_DIRECT)
        Q = colmajor_dev(q0 * 2.0 ** e)
        Qt = torch.zeros_like(Q)
        with pytest.raises(lib.RafeastError) as ei:
            lib.rafeast_filter(h, prm, Q, None, Qt)
        assert ei.value.code == lib.RAFEAST_ERR_COCG_BREAKDOWN
    finally:
        lib.rafeast_destroy(h)


@pytest.mark.parametrize("kind", ["knn", "rgg"])
def test_a_stopped_column_leaves_its_neighbours_and_result_alone(lib, kind):
    """A constant column is an eigenvector: it stops at step 1, and near the end
    of the range the scale of its last vector overflows. Its result, and those of
    the columns that go on beside it in the same 16 bytes, are those of a dense
    solve; on both routes of the neighbour sums. Tolerance: that of
    test_fixed_point_sums_against_dense."""
    import torch
    lap = _dense_graph(kind)
    A, n, (lo, hi), m0, nc = lap.scipy().toarray(), lap.n, (0.1, 4.1), 6, 4
    q = OF.random_start(n, m0, 1)
    q[:, 1] = n ** -0.5
    q[:, 4] = n ** -0.5
    z, w = OQ.nodes(lo, hi, nc, 1.0)
    exp = sum((wj * np.linalg.solve(zj * np.eye(n) - A, q)).real for zj, wj in zip(z, w))
    h = lib.rafeast_create(lap.row_ptr, lap.col_idx, lap.values, lap.shift)
    try:
        for values_free in (0, 1):
            lib.rafeast_set_option(h, lib.RAFEAST_OPT_VALUES_FREE, values_free)
            prm = lib.make_params(lo, hi, m0, nc, 1.0, 1e-12, 1e-10, 1, 2000, lib.RAFEAST_FP64,
                                  lib.RAFEAST_FORM_DIRECT)
            for e in (0, 480, 492, 494, 496, 498):
                x = 2.0 ** e
                Q = colmajor_dev(q * x)
                Qt = torch.zeros_like(Q)
                info = lib.rafeast_filter(h, prm, Q, None, Qt)
                err = np.linalg.norm(from_colmajor(Qt) / x - exp, axis=0)
                per_step = 4.0 * 2.0 ** -52 * np.abs(A).sum(0).max() * (info.cocg_max_last + 1)
                assert np.max(err) <= np.sum(np.abs(w) * (1e-12 + per_step / z.imag) / z.imag), e
    finally:
        lib.rafeast_destroy(h)


def _star_and_circulant(n):
    """One vertex joined to all of a circulant graph of eight neighbours a vertex."""
    k, t = n - 1, np.arange(1, n)
    i = np.concatenate([np.zeros(k, int)] + [t] * 4)
    j = np.concatenate([t] + [1 + (t - 1 + d) % k for d in (1, 2, 3, 5)])
    return G._from_edges(n, i, j, 0.2, "star")


def _steps_in_extended_precision(lap, q, z, w, steps):
    """Quadrature sum after `steps` Lanczos steps per column, u_{k+1} =
    L u_k - alpha_k u_k - g_k u_{k-1} without scaling, in long double."""
    A, ld = lap.scipy(), np.longdouble
    row = np.repeat(np.arange(lap.n), np.diff(A.indptr))
    off = row != A.indices
    first = np.concatenate([[0], np.cumsum(np.bincount(row[off]))[:-1]])
    col, deg = A.indices[off], np.bincount(row[off])[:, None].astype(ld)
    u, up, rr_prev = q.astype(ld), np.zeros_like(q, ld), np.ones(q.shape[1], ld)
    zz = (z - lap.shift).astype(np.clongdouble)[:, None]
    rho, dinv = np.ones((len(z), q.shape[1]), np.clongdouble), np.zeros((len(z), q.shape[1]), np.clongdouble)
    us, ts, es = [], [], []
    for k in range(steps):
        lu = deg * u - np.add.reduceat(u[col], first, axis=0)
        rr = (u * u).sum(0)
        alpha, g = (u * lu).sum(0) / rr, (rr / rr_prev if k else np.zeros_like(rr))
        t = g * dinv
        dinv = 1 / (zz - alpha - t)
        eta = rho * dinv
        us.append(u), ts.append(t), es.append(w[:, None] * eta)
        rho, rr_prev = eta, rr
        u, up = lu - alpha * u - g * up, u
    out, e, tn = np.zeros_like(q, ld), 0, 0
    for k in reversed(range(steps)):
        e, tn = es[k] + tn * e, ts[k]
        out += e.real.sum(0) * us[k]
    return out


def test_fixed_point_sums_are_as_accurate_as_fp64_sums(lib):
    """Just inside the rule for fixed point (n max deg / mean deg = 36,000 of
    41,000), on columns that stay off the vertex of the greatest degree, where a
    unit made from more than the step's own norms is coarse. After three steps the
    error against long double is compared with that of the FP64 sums
    (RAFEAST_OPT_VALUES_FREE = 1): rounding to units adds at most an error of the
    same size, sqrt(2) in the geometric mean over 96 columns."""
    import torch
    n, m0, nc, steps, (lo, hi) = 600, 96, 4, 3, (4.0, 12.0)
    lap = _star_and_circulant(n)
    q = np.random.default_rng(0).standard_normal((n, m0))
    q[0] = 0.0
    q[1:] -= q[1:].mean(0)
    q /= np.linalg.norm(q, axis=0)
    z, w = OQ.nodes(lo, hi, nc, 1.0)
    exp = _steps_in_extended_precision(lap, q, z, w, steps)
    h = lib.rafeast_create(lap.row_ptr, lap.col_idx, lap.values, lap.shift)
    try:
        err = []
        for values_free in (0, 1):
            lib.rafeast_set_option(h, lib.RAFEAST_OPT_VALUES_FREE, values_free)
            prm = lib.make_params(lo, hi, m0, nc, 1.0, 0.0, 1e-10, 1, steps, lib.RAFEAST_FP64,
                                  lib.RAFEAST_FORM_DIRECT)
            Q = colmajor_dev(q)
            Qt = torch.zeros_like(Q)
            lib.rafeast_filter(h, prm, Q, None, Qt)
            err.append(np.sqrt(((from_colmajor(Qt) - exp) ** 2).sum(0)).astype(float))
    finally:
        lib.rafeast_destroy(h)
    assert np.exp(np.mean(np.log(err[0] / err[1]))) <= np.sqrt(2.0)


@pytest.mark.parametrize("kind,fixed", [("knn", True), ("rgg", True), ("complete", True), ("hub", False),
                                        (500, True), (636, True), (660, False), ("grid", False)])
def test_which_neighbour_sums_run(lib, kind, fixed):
    """Fixed point for eight or more neighbours a row and n max deg / mean deg <=
    41,000 (a number: that many vertices of a star and circulant, 25,000, 40,500
    and 43,700), never for read values, in float or in a filter of another form."""
    import torch
    lap = G.grid2d(20, 23, shift=0.3) if kind == "grid" else \
        _star_and_circulant(kind) if isinstance(kind, int) else _dense_graph(kind)
    h = lib.rafeast_create(lap.row_ptr, lap.col_idx, lap.values, lap.shift)
    try:
        for prec, values_free, update, exp in ((lib.RAFEAST_FP64, 0, 0, fixed), (lib.RAFEAST_FP64, 1, 0, False),
                                               (lib.RAFEAST_MIXED, 0, 0, False), (lib.RAFEAST_FP64, 0, 2, False)):
            lib.rafeast_set_option(h, lib.RAFEAST_OPT_VALUES_FREE, values_free)
            lib.rafeast_set_option(h, lib.RAFEAST_OPT_UPDATE, update)
            prm = lib.make_params(0.31, 4.0, 6, 2, 1.0, 1e-2, 1e-10, 1, 20, prec, lib.RAFEAST_FORM_DIRECT)
            Q = colmajor_dev(OF.random_start(lap.n, 6, 1))
            lib.rafeast_filter(h, prm, Q, None, torch.zeros_like(Q))
            p = lib.rafeast_profile(h, reset=False)
            assert p["fixed_sums"] is exp and (update or p["update_shape"] == 0), (prec, values_free, update)
    finally:
        lib.rafeast_destroy(h)


@pytest.mark.parametrize("m0,nc", [(6, 2), (69, 4)])
@pytest.mark.parametrize("n", [500, 636])
def test_fixed_point_sums_with_a_hub_against_dense(lib, monkeypatch, n, m0, nc):
    """test_fixed_point_sums_against_dense on graphs with one vertex joined to all
    that take the fixed-point route (its own is over the rule's line)."""
    import test_gpu_lanczos as here
    monkeypatch.setattr(here, "_dense_graph", lambda kind: _star_and_circulant(n))
    here.test_fixed_point_sums_against_dense(lib, "star", m0, nc)
