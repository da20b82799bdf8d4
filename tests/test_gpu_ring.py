"""The device memory that rings of Lanczos vectors take, leave and give back.
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
    rounding (2^2 eps ||A|| of matrix error per step over 2^7 steps, doubled by the
    two folds' roundings; ||A||_1 <= 12.3)."""
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


def test_alternating_widths_keep_the_ring(lib, cube):
    """A narrow filter takes the slabs of a wide one: the free memory stays as it is
    from the second call on (workspaces grow with the widest)."""
    _, run = cube
    left = []
    for m0 in (24, 96, 24, 96, 24):
        run(0, m0, 40)
        left.append(_free())
    assert len(set(left[1:])) == 1


