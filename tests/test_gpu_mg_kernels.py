"""Restriction and coarse operator at the edges of their kernels: 1 to 32 test
vectors (groups of 8 in the restriction; rows padded to 4 and 4, 8, 9, 12 or
more chunks per thread in the coarse operator), aggregates of 16 sites (half a
warp) and of 256. Bounds as in test_gpu_mg.py: FP16 entries of P and D_c."""
import numpy as np
import pytest

import paper_1710_07041_gb300 as dd
import synth
from gpu_common import Setup, relerr
from oracle.twolevel import TwoLevel

pytestmark = pytest.mark.gpu

SMALL, WIDE = ((4, 4, 4, 4), (2, 2, 2, 2)), ((8, 8, 8, 8), (4, 4, 4, 4))


@pytest.mark.parametrize("shape,n", [(SMALL, n) for n in (1, 7, 8, 9, 15, 16, 17, 19, 32)] + [(WIDE, 16)])
def test_restriction_and_coarse_operator(shape, n):
    dims, block = shape
    s = Setup(dims, block, eps=0.3, n_stout=1, c_sw=1.0, m0=-0.05, prec=dd.F32, seed=93)
    tv = np.stack([synth.gaussian_spinor(s.V, 940 + k) for k in range(n)])
    mg = dd.Multigrid(s.op, tv, setup_iters=0, coarse_max_iter=4, coarse_tol=0.0, sweeps=1, mr_steps=1)
    tl = TwoLevel(s.ref, block, tv)
    rf = s.lat.to_field(synth.gaussian_spinor(s.V, 931), dd.F32)
    c = mg.new_coarse()
    mg.restrict(rf, c)
    got = dd.Multigrid.coarse_to_numpy(c, tl.nagg, tl.N)
    assert relerr(got, tl.restrict(s.lat.from_field(rf, dd.F32))) <= 2e-3
    cc = synth.gaussian(tl.nagg * 2 * tl.N, 932).reshape(tl.nagg, 2, tl.N).astype(np.complex64)
    mg.coarse_apply(dd.Multigrid.coarse_from_numpy(cc), c)
    assert relerr(dd.Multigrid.coarse_to_numpy(c, tl.nagg, tl.N), tl.coarse_apply(cc)) <= 2e-3
    mg.close()
    s.close()
