"""The packed Schwarz kernel (4^4 and 8 x 4^3 blocks, 32- and 16-bit storage)
where its bookkeeping can go wrong: lattices of two blocks per direction (both
neighbours of a block are the same one, every hop across the edge), an
elongated one with the other extents minimal, with and without the
antiperiodic sign, from x = 0 and from a given x (whose first residual b - D x
is a launch of its own), one right-hand side and several sharing a CTA, one
and two sweeps, 0 to 3 MR steps. Each against the FP64 oracle; and the
general kernel on the same operator fields.

Bounds (relative L2): those of test_gpu_sap.py, a few unit roundoffs of the
storage (b and the operator rounded once, x once per sweep)."""
import os
import subprocess
import sys

import numpy as np
import pytest

import paper_1710_07041_gb300 as dd
import synth
from gpu_common import Setup, relerr

pytestmark = pytest.mark.gpu

TOL = {dd.F32: 5e-7, dd.F16: 1.5e-3, dd.BF16: 1.2e-2, dd.F16N: 1e-3}
CASES = [((8, 8, 8, 8), (4, 4, 4, 4), True, 2, 3), ((8, 8, 8, 24), (4, 4, 4, 4), False, 1, 1),
         ((16, 8, 8, 8), (8, 4, 4, 4), True, 2, 2), ((16, 8, 24, 8), (8, 4, 4, 4), False, 1, 0)]


@pytest.mark.parametrize("prec", [dd.F32, dd.F16, dd.BF16, dd.F16N])
@pytest.mark.parametrize("dims,block,anti,sweeps,nmr", CASES)
@pytest.mark.parametrize("guess", [False, True])
def test_packed_kernel(prec, dims, block, anti, sweeps, nmr, guess):
    s = Setup(dims, block, eps=0.3, n_stout=1, c_sw=1.7, m0=-0.02, prec=prec, seed=31, antiperiodic=anti)
    n = 3
    b = np.stack([synth.gaussian_spinor(s.V, 40 + r) for r in range(n)])
    x0 = np.stack([0.1 * synth.gaussian_spinor(s.V, 50 + r) for r in range(n)])
    fb = s.lat.to_field(b, prec)
    start = s.lat.from_field(s.lat.to_field(x0, prec), prec, n)   # x as stored
    for tile in (1, 2):
        fx = s.lat.to_field(x0, prec)
        s.op.sap_smooth(fb, fx, sweeps, nmr, nrhs=n, x_is_zero=not guess, rhs_tile=tile)
        got = s.lat.from_field(fx, prec, n)
        for r in range(n):
            want = s.ref.sap(block, b[r], sweeps, nmr, x0=start[r] if guess else None)
            assert relerr(got[r], want) <= TOL[prec], (tile, r)
    dd.device_status()   # no staging wait expired
    s.close()


CHILD = r'''
import sys
import numpy as np
import paper_1710_07041_gb300 as dd
import synth
from gpu_common import Setup
out = {}
for prec in (dd.F32, dd.F16):
    for dims, block in (((8, 8, 8, 16), (4, 4, 4, 4)), ((16, 8, 8, 8), (8, 4, 4, 4))):
        s = Setup(dims, block, eps=0.3, n_stout=1, c_sw=1.7, m0=-0.02, prec=prec, seed=33)
        fb, fx = s.lat.to_field(synth.gaussian_spinor(s.V, 34), prec), s.lat.new_field(prec)
        s.op.sap_smooth(fb, fx, 2, 3)
        out["%d_%d" % (prec, block[0])] = s.lat.from_field(fx, prec)
        s.close()
np.savez(sys.argv[1], **out)
'''


def test_packed_kernel_agrees_with_the_recomputing_form(tmp_path):
    """DD_SAP_INCR=0 takes the general kernel, which forms b - D x in every
    phase, on the same operator fields: the two differ by rounding only (twice
    the bound against the oracle)."""
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    got = []
    for incr in ("1", "0"):
        env = dict(os.environ, DD_SAP_INCR=incr,
                   PYTHONPATH=os.pathsep.join([root, os.path.join(root, "tests"), os.environ.get("PYTHONPATH", "")]))
        f = str(tmp_path / f"x{incr}.npz")
        p = subprocess.run([sys.executable, "-c", CHILD, f], cwd=root, env=env, capture_output=True, text=True,
                           timeout=600)
        assert p.returncode == 0, p.stdout[-2000:] + p.stderr[-4000:]
        got.append(dict(np.load(f)))
    assert len(got[0]) == 4
    for k in got[0]:
        assert relerr(got[0][k], got[1][k]) <= 2 * TOL[int(k.split("_")[0])], k
