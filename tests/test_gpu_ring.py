"""The ring of Lanczos vectors when it is smaller than the solve: its steps are
folded into the quadrature sum and one direction per node, and its slots are used
again (RAFEAST_OPT_RING_SLOTS caps the slots). And the device memory that rings
take, leave and give back.

Slots: 4 folds every two steps, 7 every four (an odd count, so slots and steps go
out of phase), 20 after 16 steps and more; node counts reach each instance of the
folding pass (1, 2, up to 4 and two or three passes), in both precisions.
Tolerances are those of test_gpu_lanczos.py: 2^2 eps ||A|| of matrix error per
step, here over at most 2^7 steps, which the folds (two more roundings of a value
per fold and node) at most double.
"""
import numpy as np
import pytest

from gpu_util import colmajor_dev, from_colmajor
from oracle import feast as OF
from oracle import quadrature as OQ
from workloads import graphs as G

pytestmark = pytest.mark.gpu

GIB = 1 << 30


def _filter(lib, h, q, prm):
    import torch
    Q = colmajor_dev(q)
    Qt = torch.zeros_like(Q)
    info = lib.rafeast_filter(h, prm, Q, None, Qt)
    return from_colmajor(Qt), info


@pytest.mark.parametrize("slots", [4, 7, 20])
@pytest.mark.parametrize("steps", [5, 33, 70])
@pytest.mark.parametrize("m0,nc", [(1, 1), (5, 2), (46, 3), (80, 4), (17, 8), (97, 12)])
def test_folded_steps_match_oracle(lib, m0, nc, steps, slots):
    lap = G.grid2d(37, 41, shift=0.3)
    A, (lo, hi) = lap.scipy(), (0.31, 0.6)
    q0 = OF.random_start(lap.n, m0, 1)
    z, w = OQ.nodes(lo, hi, nc, 1.0)
    exp, _ = OF.filter_apply(A, q0, z, w, 0.0, steps, "direct")
    bound = 2.0 ** 10 * OF.one_norm(A) * np.sum(np.abs(w) / z.imag ** 2)
    h = lib.rafeast_create(lap.row_ptr, lap.col_idx, lap.values, lap.shift)
    try:
        lib.rafeast_set_option(h, lib.RAFEAST_OPT_RING_SLOTS, slots)
        for prec, tiled, eps in ((lib.RAFEAST_FP64, 1, 2.0 ** -52), (lib.RAFEAST_MIXED, 1, 2.0 ** -23),
                                 (lib.RAFEAST_MIXED, 2, 2.0 ** -23)):
            lib.rafeast_set_option(h, lib.RAFEAST_OPT_TILED, tiled)
            prm = lib.make_params(lo, hi, m0, nc, 1.0, 0.0, 1e-10, 1, steps, prec, lib.RAFEAST_FORM_DIRECT)
            got, info = _filter(lib, h, q0, prm)
            assert info.cocg_min_last == info.cocg_max_last == steps
            assert np.max(np.linalg.norm(got - exp, axis=0)) <= bound * eps, (prec, tiled)
    finally:
        lib.rafeast_destroy(h)


@pytest.mark.parametrize("slots", [4, 7, 20])
@pytest.mark.parametrize("m0,nc", [(7, 1), (9, 2), (46, 4), (21, 12)])
@pytest.mark.parametrize("kind", ["grid", "rgg", "weighted"])
def test_columns_that_stop_in_different_folds(lib, kind, m0, nc, slots):
    """FP64 solves to 1e-12 against a dense solve: columns and nodes stop many
    folds apart (a zero column and a constant one, which is an eigenvector, at once; a
    unit vector; random ones), on FP64 sums, fixed-point sums and read values.
    Tolerance as in test_fixed_point_sums_against_dense, steps counted twice."""
    if kind == "grid":
        lap = G.grid2d(23, 29, shift=0.2)
    else:
        lap = G.rgg2d(700, seed=3, shift=0.2)
    A, n, (lo, hi) = lap.scipy().tocsr(), lap.n, (0.1, 4.1)
    val = lap.values
    if kind == "weighted":
        rng = np.random.default_rng(1)
        s = 0.5 + rng.random(n)
        A = A.multiply(np.outer(s, s)).tocsr()
        A.sort_indices()
        val = A.data
        row_ptr, col_idx, shift = A.indptr.astype(np.int32), A.indices.astype(np.int32), 0.0
    else:
        row_ptr, col_idx, shift = lap.row_ptr, lap.col_idx, lap.shift
    A = A.toarray()
    q = OF.random_start(n, m0, 1)
    q[:, 0] = 0.0
    q[:, 1] = n ** -0.5
    q[:, 2] = 0.0
    q[n // 3, 2] = 1.0
    z, w = OQ.nodes(lo, hi, nc, 1.0)
    exp = sum((wj * np.linalg.solve(zj * np.eye(n) - A, q)).real for zj, wj in zip(z, w))
    h = lib.rafeast_create(row_ptr, col_idx, val, shift)
    try:
        lib.rafeast_set_option(h, lib.RAFEAST_OPT_RING_SLOTS, slots)
        prm = lib.make_params(lo, hi, m0, nc, 1.0, 1e-12, 1e-10, 1, 3000, lib.RAFEAST_FP64,
                              lib.RAFEAST_FORM_DIRECT)
        got, info = _filter(lib, h, q, prm)
        assert info.cocg_max_last < 3000 and np.all(got[:, 0] == 0.0)
        per_step = 8.0 * 2.0 ** -52 * np.abs(A).sum(0).max() * (info.cocg_max_last + 1)
        tol = np.sum(np.abs(w) * (1e-12 + per_step / z.imag) / z.imag)
        assert np.max(np.linalg.norm(got - exp, axis=0)) <= tol
        # float: the tiled product makes the same vectors whatever the ring, so the
        # filters differ by the folds' roundings
        if kind == "grid":
            lib.rafeast_set_option(h, lib.RAFEAST_OPT_TILED, 2)
            prm = lib.make_params(lo, hi, m0, nc, 1.0, 1e-3, 1e-10, 1, 60, lib.RAFEAST_MIXED,
                                  lib.RAFEAST_FORM_DIRECT)
            out = []
            for s in (0, slots):
                lib.rafeast_set_option(h, lib.RAFEAST_OPT_RING_SLOTS, s)
                out.append(_filter(lib, h, q, prm)[0])
            bound = 2.0 ** 10 * 2.0 ** -23 * np.abs(A).sum(0).max() * np.sum(np.abs(w) / z.imag ** 2)
            assert np.max(np.linalg.norm(out[0] - out[1], axis=0)) <= bound
    finally:
        lib.rafeast_destroy(h)


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
def test_batched_folds(lib, prec):
    """As test_batched_filter_matches_one_at_a_time, with rings of 4, 7 and 20
    slots for the batch (the first handle's option) against rings that hold all."""
    shapes, m0s = [(5, 7), (20, 23), (37, 41), (90, 101)], [3, 8, 17, 30]
    p = lib.RAFEAST_FP64 if prec == "fp64" else lib.RAFEAST_MIXED
    laps = [G.grid2d(a, b, shift=0.1 * (t + 1)) for t, (a, b) in enumerate(shapes)]
    prms = [lib.make_params(0.05, 0.1 * (t + 1) + 0.3, m, 3, 0.5, 1e-3, 0.0, 2, 40 + 13 * t, p,
                            lib.RAFEAST_FORM_CORRECTION, lib.RAFEAST_START_RANDOM, 5)
            for t, m in enumerate(m0s)]
    hs = [lib.rafeast_create(x.row_ptr, x.col_idx, x.values, x.shift) for x in laps]
    try:
        ref = [np.zeros(m) for m in m0s]
        _, mf0, _ = lib.rafeast_solve_batched(hs, prms, ref)
        eps = 2.0 ** -52 if prec == "fp64" else 2.0 ** -23
        for slots in (4, 7, 20):
            lib.rafeast_set_option(hs[0], lib.RAFEAST_OPT_RING_SLOTS, slots)
            ev = [np.zeros(m) for m in m0s]
            _, mf, _ = lib.rafeast_solve_batched(hs, prms, ev)
            assert list(mf) == list(mf0)
            for a, b in zip(ev, ref):
                assert np.max(np.abs(np.sort(a) - np.sort(b))) <= 2.0 ** 10 * eps * 8.5
    finally:
        for h in hs:
            lib.rafeast_destroy(h)


def test_option_values(lib):
    lap = G.grid2d(5, 7, shift=0.3)
    h = lib.rafeast_create(lap.row_ptr, lap.col_idx, lap.values, lap.shift)
    try:
        for bad in (-1, 1, 3, (1 << 20) + 1):
            with pytest.raises(lib.RafeastError):
                lib.rafeast_set_option(h, lib.RAFEAST_OPT_RING_SLOTS, bad)
        lib.rafeast_set_option(h, lib.RAFEAST_OPT_RING_SLOTS, 0)
    finally:
        lib.rafeast_destroy(h)


# ---- device memory: the 50 x 50 x 50 grid with 96 float columns has slots of 46 MiB,
# slabs of a gibibyte (22 slots) and, after 100 steps, five of them ---------------

def _free():
    import torch
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    return torch.cuda.mem_get_info()[0]


def _hold_all_but(rest):
    import torch
    return torch.empty(_free() - rest, dtype=torch.uint8, device="cuda")


@pytest.fixture
def cube(lib):
    import torch
    lap = G.grid3d(50, 50, 50, 0.3)
    hs = [lib.rafeast_create(lap.row_ptr, lap.col_idx, lap.values, lap.shift) for _ in range(2)]
    q = colmajor_dev(OF.random_start(lap.n, 96, 1))
    out = [torch.zeros_like(q) for _ in hs]

    def run(t, m0=96, cap=100):
        prm = lib.make_params(0.31, 0.6, m0, 1, 1.0, 0.0, 1e-10, 1, cap, lib.RAFEAST_MIXED,
                              lib.RAFEAST_FORM_DIRECT)
        lib.rafeast_filter(hs[t], prm, q, None, out[t])
        return out[t]
    yield hs, run
    for h in hs:
        lib.rafeast_destroy(h)


def test_ring_leaves_memory_to_others(lib, cube):
    """With 6 GiB free a ring that took all it could use would leave a few hundred
    megabytes; one that keeps a sixteenth of the device free takes the gibibyte
    that it cannot do without, of about 1.6 with the filter's blocks."""
    _, run = cube
    hold = _hold_all_but(6 * GIB)
    run(0)
    left = _free()
    del hold
    assert left >= 4 * GIB


def test_idle_rings_are_given_to_another_handle(lib, cube):
    """The second handle's blocks and smallest ring (0.6 GiB) do not fit the 0.35
    that are free: the first handle's idle ring makes room, and comes back for the
    first handle's next filter. Both filters of the same block are the same up to
    the folds' roundings (bound of test_folded_steps_match_oracle, ||A||_1 <= 12.3)."""
    _, run = cube
    first = run(0).clone()
    hold = _hold_all_but(int(0.35 * GIB))
    second = run(1)
    del hold
    z, w = OQ.nodes(0.31, 0.6, 1, 1.0)
    bound = 2.0 ** 10 * 2.0 ** -23 * 12.3 * np.sum(np.abs(w) / z.imag ** 2)
    assert float((first - second).norm(dim=1).max()) <= bound
    _free()
    again = run(0)
    assert float((first - again).norm(dim=1).max()) <= bound


def test_filter_runs_once_more_with_the_smallest_ring(lib, cube):
    """1.15 GiB free: the blocks of 0.4 fit, a slab of a gibibyte beside them does
    not, the smallest ring and its directions (0.3) do."""
    _, run = cube
    first = run(0).clone()
    hold = _hold_all_but(int(1.15 * GIB))
    lib.rafeast_set_option(cube[0][0], lib.RAFEAST_OPT_RING_SLOTS, 0)  # (its ring: to the device)
    hold2 = _hold_all_but(int(1.15 * GIB))
    second = run(1)
    del hold, hold2
    z, w = OQ.nodes(0.31, 0.6, 1, 1.0)
    bound = 2.0 ** 10 * 2.0 ** -23 * 12.3 * np.sum(np.abs(w) / z.imag ** 2)
    assert float((first - second).norm(dim=1).max()) <= bound


def test_alternating_widths_keep_the_ring(lib, cube):
    """A narrow filter takes the slabs of a wide one: the free memory stays as it is
    from the second call on (workspaces grow with the widest)."""
    _, run = cube
    left = []
    for m0 in (24, 96, 24, 96, 24):
        run(0, m0, 40)
        left.append(_free())
    assert len(set(left[1:])) == 1


def test_setting_the_option_gives_the_ring_back(lib, cube):
    hs, run = cube
    run(0)
    before = _free()
    lib.rafeast_set_option(hs[0], lib.RAFEAST_OPT_RING_SLOTS, 0)
    assert _free() - before >= 4 * GIB


def test_batch_runs_once_more_with_the_smallest_rings(lib, cube):
    """The batch's workspaces are there from a first run; with its rings given back
    and 0.9 GiB free no slab of a gibibyte can be had, the smallest rings of both
    handles (0.2 and 0.1 of directions each) can."""
    hs, _ = cube
    prm = [lib.make_params(0.25, 0.4, 96, 1, 1.0, 1e-2, 0.0, 2, 40, lib.RAFEAST_MIXED,
                           lib.RAFEAST_FORM_CORRECTION, lib.RAFEAST_START_RANDOM, 5)] * 2
    ref, ev = [[np.zeros(96) for _ in hs] for _ in range(2)]
    lib.rafeast_solve_batched(hs, prm, ref)
    for h in hs:
        lib.rafeast_set_option(h, lib.RAFEAST_OPT_RING_SLOTS, 0)
    hold = _hold_all_but(int(0.9 * GIB))
    lib.rafeast_solve_batched(hs, prm, ev)
    del hold
    for a, b in zip(ev, ref):
        assert np.max(np.abs(np.sort(a) - np.sort(b))) <= 2.0 ** 10 * 2.0 ** -23 * 12.3
