"""Memory that the library keeps between calls is given back where an
allocation needs it: the set-up of an operator beside kept work fields, and the
work fields of a smoother call beside a kept solver workspace (without them the
call takes the general kernel, whose bits differ). Where the work fields do not
fit for all right-hand sides the call takes as many at a time as they do for.

Other memory of the device is taken by a filler, all but MARGIN bytes."""
import numpy as np
import pytest
import torch

import paper_1710_07041_gb300 as dd
import synth

pytestmark = pytest.mark.gpu

MARGIN = 600 << 20


def fill():
    """Takes the free device memory but MARGIN."""
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    held = []
    while (free := torch.cuda.mem_get_info()[0]) > MARGIN + (64 << 20):
        held.append(torch.empty(min(free - MARGIN, 32 << 30), dtype=torch.uint8, device="cuda"))
    return held


def unit_gauge(lat):
    return dd.Gauge(lat, np.tile(np.eye(3, dtype=np.complex128), (lat.V, 4, 1, 1)))


def small_op():
    lat = dd.Lattice((32, 16, 16, 16), (4, 4, 4, 4))
    return lat, dd.Op(dd.Gauge(lat, synth.gauge((32, 16, 16, 16), 0.25, 0, 0.1, 3)), 1.0, 0.1, dd.F32)


def keep_workspace(lat, op):
    """A solve, which leaves its workspace in the cache (2.6 GB)."""
    op.solve(np.stack([synth.gaussian_spinor(lat.V, 81)] * 2), tol=1e-6, restart=32, sweeps=2, mr_steps=3)


def test_setup_takes_back_what_is_kept():
    assert dd.lib().dd_release_workspace() == 0
    lat, op = small_op()
    n = 16
    b, x = lat.new_field(dd.F32, n), lat.new_field(dd.F32, n)
    op.sap_smooth(b, x, 1, 1, nrhs=n)   # leaves its work fields in the pool (0.4 GB)
    keep_workspace(lat, op)
    big = dd.Lattice((32, 32, 16, 16), (4, 4, 4, 4))
    held = fill()
    try:
        other = dd.Op(unit_gauge(big), 1.0, 0.1, dd.F32)   # 1.1 GB
        mg = dd.Multigrid(other, np.ones((2, big.V, 4, 3), dtype=np.complex128), setup_iters=0, sweeps=1, mr_steps=1)
        mg.close()
        other.close()
    finally:
        del held
        torch.cuda.empty_cache()
    op.close()


def test_work_fields_take_back_a_kept_workspace():
    assert dd.lib().dd_release_workspace() == 0
    lat, op = small_op()
    n = 40   # work fields: 40 x 25 MB
    b = lat.to_field(np.stack([synth.gaussian_spinor(lat.V, 80)] * n), dd.F32)
    x, y = lat.new_field(dd.F32, n), lat.new_field(dd.F32, n)
    op.sap_smooth(b, x, 2, 3, nrhs=n)
    torch.cuda.synchronize()
    assert dd.lib().dd_release_workspace() == 0
    keep_workspace(lat, op)
    held = fill()
    try:
        op.sap_smooth(b, y, 2, 3, nrhs=n)
        torch.cuda.synchronize()
    finally:
        del held
        torch.cuda.empty_cache()
    assert torch.equal(x, y)
    op.close()


@pytest.mark.parametrize("guess", [False, True])
@pytest.mark.parametrize("several", [False, True])
def test_work_fields_for_some_right_hand_sides_at_a_time(guess, several):
    assert dd.lib().dd_release_workspace() == 0
    lat, op = small_op()
    n = 64   # work fields: 64 x 25 MB, from a given x 64 x 38 MB
    b = lat.to_field(np.stack([synth.gaussian_spinor(lat.V, 82)] * n), dd.F32)
    x, y = lat.new_field(dd.F32, n), lat.new_field(dd.F32, n)

    def smooth(x):
        if several:
            h = b.numel() // 2
            dd.sap_smooth_multi([(op, b[:h], x[:h], n // 2), (op, b[h:], x[h:], n // 2)], 2, 3, x_is_zero=not guess)
        else:
            op.sap_smooth(b, x, 2, 3, nrhs=n, x_is_zero=not guess)
        torch.cuda.synchronize()

    smooth(x)
    assert dd.lib().dd_release_workspace() == 0
    held = fill()
    try:
        smooth(y)
    finally:
        del held
        torch.cuda.empty_cache()
    assert torch.equal(x, y)
    op.close()
