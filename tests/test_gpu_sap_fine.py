"""The FP64 small-block Schwarz kernel (blocks of 16 and 32 sites) against the
FP64 oracle: both sizes, two blocks per direction and an elongated lattice,
with and without the antiperiodic sign, from x = 0 and from a given x (whose
first sweep forms b - D x from x), several right-hand sides with one and two
per CTA, 0 to 3 MR steps. Bound: rounding order only, as in test_gpu_sap.py."""
import numpy as np
import pytest

import paper_1710_07041_gb300 as dd
import synth
from gpu_common import Setup, relerr

pytestmark = pytest.mark.gpu

CASES = [((4, 4, 4, 4), (2, 2, 2, 2), True, 3), ((4, 4, 12, 8), (2, 2, 2, 2), False, 1),
         ((8, 4, 4, 4), (4, 2, 2, 2), True, 2), ((4, 4, 4, 16), (2, 2, 2, 4), False, 0)]


@pytest.mark.parametrize("dims,block,anti,nmr", CASES)
@pytest.mark.parametrize("guess", [False, True])
def test_small_block_kernel(dims, block, anti, nmr, guess):
    s = Setup(dims, block, eps=0.3, n_stout=1, c_sw=1.7, m0=-0.02, prec=dd.F64, seed=61, antiperiodic=anti)
    n = 3
    b = np.stack([synth.gaussian_spinor(s.V, 62 + r) for r in range(n)])
    x0 = np.stack([0.1 * synth.gaussian_spinor(s.V, 72 + r) for r in range(n)])
    fb = s.lat.to_field(b, dd.F64)
    for tile in (1, 2):
        fx = s.lat.to_field(x0, dd.F64)
        s.op.sap_smooth(fb, fx, 2, nmr, nrhs=n, x_is_zero=not guess, rhs_tile=tile)
        got = s.lat.from_field(fx, dd.F64, n)
        for r in range(n):
            want = s.ref.sap(block, b[r], 2, nmr, x0=x0[r] if guess else None)
            assert relerr(got[r], want) <= 1e-12, (tile, r)
    s.close()


def test_small_block_kernel_several_lattices():
    """One launch over two lattices equals the single launches bit for bit."""
    import torch
    setups, items, singles = [], [], []
    for dims, nrhs, seed in (((4, 4, 4, 4), 2, 63), ((4, 4, 8, 4), 1, 64)):
        s = Setup(dims, (2, 2, 2, 2), prec=dd.F64, seed=seed)
        b = np.stack([synth.gaussian_spinor(s.V, seed + 10 + r) for r in range(nrhs)])
        fb, fx = s.lat.to_field(b, dd.F64), s.lat.new_field(dd.F64, nrhs)
        s.op.sap_smooth(fb, fx, 2, 3, nrhs=nrhs)
        setups.append(s)
        singles.append(fx)
        items.append((s.op, fb, s.lat.new_field(dd.F64, nrhs), nrhs))
    dd.sap_smooth_multi(items, 2, 3)
    torch.cuda.synchronize()
    for single, (_, _, fx, _) in zip(singles, items):
        assert torch.equal(fx, single)
    for s in setups:
        s.close()


@pytest.mark.parametrize("dims,block,anti", [((4, 4, 4, 4), (2, 2, 2, 2), True), ((4, 4, 4, 4), (2, 2, 2, 2), False),
                                             ((4, 12, 4, 4), (2, 2, 2, 2), True), ((8, 8, 4, 4), (4, 2, 2, 2), True)])
def test_small_lattice_operator(dims, block, anti):
    """The FP64 Dslash of the smallest lattices (up to 1024 sites): each of
    three right-hand sides against the oracle (bound: rounding order, as in
    test_gpu_operator.py), and the same bits alone."""
    s = Setup(dims, block, eps=0.3, n_stout=1, c_sw=1.7, m0=-0.02, prec=dd.F64, seed=65, antiperiodic=anti)
    psi = np.stack([synth.gaussian_spinor(s.V, 66 + r) for r in range(3)])
    out = s.lat.new_field(dd.F64, 3)
    s.op.apply_D(dd.F64, s.lat.to_field(psi, dd.F64), out, nrhs=3)
    got = s.lat.from_field(out, dd.F64, 3)
    for r in range(3):
        assert relerr(got[r], s.ref.apply(psi[r])) <= 1e-13, r
        one = s.lat.new_field(dd.F64)
        s.op.apply_D(dd.F64, s.lat.to_field(psi[r], dd.F64), one)
        assert np.array_equal(s.lat.from_field(one, dd.F64), got[r])
    s.close()
