"""The default recurrence (real Lanczos) step by step on every kind of matrix: unit
grids, a reordered kNN graph, weighted Laplacians (values read) and a random
symmetric matrix with empty rows; every shape of the register-gather product that
an option can force, and every block width of the tiled one.

Twelve fixed steps against the oracle's COCG; tolerance per unit column as in
test_gpu_lanczos.py: 2^9 eps ||A|| sum_j |w_j| / Im(z_j)^2, of which twelve steps of
2^2 roundings use an eighth.
"""
import numpy as np
import pytest

from gpu_util import colmajor_dev, from_colmajor
from oracle import feast as OF
from oracle import quadrature as OQ
from test_gpu_tiled import TILED_SHAPE, _matrix

pytestmark = pytest.mark.gpu

STEPS = 12


@pytest.mark.parametrize("kind", ["grid", "knn", "weighted", "empty_rows"])
@pytest.mark.parametrize("m0,nc", [(3, 1), (17, 2), (46, 4), (80, 8), (97, 3)])
def test_forms_match_oracle_stepwise(lib, kind, m0, nc):
    import torch
    rp, ci, va, shift, A, (lo, hi) = _matrix(kind)
    q0 = OF.random_start(A.shape[0], m0, 1)
    Q = colmajor_dev(q0)
    z, w = OQ.nodes(lo, hi, nc, 1.0)
    exp, _ = OF.filter_apply(A, q0, z, w, 0.0, STEPS, "direct")
    bound = 2.0 ** 9 * OF.one_norm(A) * np.sum(np.abs(w) / z.imag ** 2)

    def check(h, prec, eps, what):
        prm = lib.make_params(lo, hi, m0, nc, 1.0, 0.0, 1e-10, 1, STEPS, prec, lib.RAFEAST_FORM_DIRECT)
        Qt = torch.full_like(Q, 7.0)
        info = lib.rafeast_filter(h, prm, Q, None, Qt)
        assert info.cocg_max_last == STEPS
        err = np.linalg.norm(from_colmajor(Qt) - exp, axis=0)
        assert np.max(err) <= bound * eps, (what, float(np.max(err)))
        return lib.rafeast_profile(h, reset=False)

    h = lib.rafeast_create(rp, ci, va, shift)
    try:
        for prec, eps in ((lib.RAFEAST_FP64, 2.0 ** -52), (lib.RAFEAST_MIXED, 2.0 ** -23)):
            lib.rafeast_set_option(h, lib.RAFEAST_OPT_TILED, 1)
            for lanes, cpl in ((4, 1), (4, 4), (8, 2), (8, 3), (16, 1), (16, 2), (32, 1)):
                lib.rafeast_set_option(h, lib.RAFEAST_OPT_LANES, lanes)
                lib.rafeast_set_option(h, lib.RAFEAST_OPT_CPL, cpl)
                p = check(h, prec, eps, (lanes, cpl))
                assert p["dots_shape"] % 10000 // 100 == lanes and p["dots_shape"] % 100 <= cpl
                assert p["fixed_sums"] is (kind == "knn" and prec == lib.RAFEAST_FP64)
        lib.rafeast_set_option(h, lib.RAFEAST_OPT_LANES, 0)
        lib.rafeast_set_option(h, lib.RAFEAST_OPT_CPL, 0)
        lib.rafeast_set_option(h, lib.RAFEAST_OPT_TILED, 2)
        for cb in (4, 5, 8, 10):
            lib.rafeast_set_option(h, lib.RAFEAST_OPT_TILE_CB, cb)
            p = check(h, lib.RAFEAST_MIXED, 2.0 ** -23, cb)
            assert (p["dots_shape"] - TILED_SHAPE) // 100 == cb
    finally:
        lib.rafeast_destroy(h)


@pytest.mark.parametrize("cb", [5, 10])
def test_cocg_forms_choose_for_themselves_at_other_widths(lib, cb):
    """Block widths that the COCG forms have no instance of leave them to the
    autotuner."""
    import torch
    rp, ci, va, shift, A, (lo, hi) = _matrix("grid")
    q0 = OF.random_start(A.shape[0], 17, 1)
    z, w = OQ.nodes(lo, hi, 4, 1.0)
    exp, _ = OF.filter_apply(A, q0, z, w, 0.0, STEPS, "direct")
    h = lib.rafeast_create(rp, ci, va, shift)
    try:
        lib.rafeast_set_option(h, lib.RAFEAST_OPT_UPDATE, 2)
        lib.rafeast_set_option(h, lib.RAFEAST_OPT_TILED, 2)
        lib.rafeast_set_option(h, lib.RAFEAST_OPT_TILE_CB, cb)
        prm = lib.make_params(lo, hi, 17, 4, 1.0, 0.0, 1e-10, 1, STEPS, lib.RAFEAST_MIXED,
                              lib.RAFEAST_FORM_DIRECT)
        Q = colmajor_dev(q0)
        Qt = torch.zeros_like(Q)
        lib.rafeast_filter(h, prm, Q, None, Qt)
        bound = 2.0 ** 9 * 2.0 ** -23 * OF.one_norm(A) * np.sum(np.abs(w) / z.imag ** 2)
        assert np.max(np.linalg.norm(from_colmajor(Qt) - exp, axis=0)) <= bound
    finally:
        lib.rafeast_destroy(h)
