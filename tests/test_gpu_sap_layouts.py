"""Every launch variant of the Schwarz kernels in 32- and 16-bit storage, forced,
on the block shapes that reach it, against the FP64 oracle (the bounds of
test_gpu_variants.py): the general kernel's layouts (operator tiles staged with
one and with two CTAs per SM, links alone staged, nothing staged), each with one
CTA per block and the persistent grid, on blocks that hand on the corrections
themselves and on 512-site ones that hand on their face flux; the packed kernel
with every number of right-hand sides per CTA. How many variants a case has is
read from the tuner's report, so that a forced one is never the default in
disguise."""
import os
import re
import subprocess
import sys

import numpy as np
import pytest

import paper_1710_07041_gb300 as dd
import synth
from gpu_common import Setup, relerr
from test_gpu_variants import SAP_TOL, forced_variant

pytestmark = pytest.mark.gpu

PRECS = [dd.F32, dd.F16, dd.BF16, dd.F16N]
# lattice, block, right-hand sides, variants
CASES = [((8, 4, 8, 8), (4, 2, 4, 4), 3, 12),     # staged once, twice per SM, not at all x 2 tiles x 2 grids
         ((16, 8, 8, 4), (8, 4, 4, 2), 3, 12),    # (FP32: links alone instead of twice)
         ((8, 8, 8, 16), (4, 4, 4, 8), 3, 4),     # face flux: one layout x 2 tiles x 2 grids
         ((16, 16, 8, 4), (8, 8, 4, 2), 3, 4),
         ((8, 8, 8, 8), (4, 4, 4, 4), 12, 5),     # packed: 1, 2, 4, 8, 12 right-hand sides per CTA
         ((16, 8, 8, 8), (8, 4, 4, 4), 12, 5)]

COUNT = r'''
import sys
import paper_1710_07041_gb300 as dd
import numpy as np
from test_gpu_sap_layouts import CASES, PRECS
for dims, block, n, _ in CASES:
    for prec in PRECS:
        lat = dd.Lattice(dims, block)
        op = dd.Op(dd.Gauge(lat, np.tile(np.eye(3, dtype=np.complex128), (lat.V, 4, 1, 1))), 0.0, 0.1, prec)
        b, x = lat.new_field(prec, n), lat.new_field(prec, n)
        op.sap_smooth(b, x, 2, 3, nrhs=n)
        op.close()
'''


def test_number_of_variants():
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    env = {k: v for k, v in os.environ.items() if not k.startswith("DD_TUNE")}
    env.update(DD_TUNE_VERBOSE="1", PYTHONPATH=os.pathsep.join([root, os.path.join(root, "tests")]))
    p = subprocess.run([sys.executable, "-c", COUNT], cwd=root, env=env, capture_output=True, text=True, timeout=600)
    assert p.returncode == 0, p.stdout[-2000:] + p.stderr[-4000:]
    got = [len(re.findall(r" v\d+=", line)) for line in p.stderr.splitlines() if line.startswith("dd tune sap")]
    assert got == [n for *_, n in CASES for _ in PRECS], p.stderr[-4000:]


@pytest.mark.parametrize("prec", PRECS)
@pytest.mark.parametrize("dims,block,n,variants", CASES)
@pytest.mark.parametrize("guess", [False, True])
def test_forced_variants(prec, dims, block, n, variants, guess):
    """Two sweeps of three steps; from a given x the choice is not tuned and the
    default variant runs."""
    s = Setup(dims, block, eps=0.3, n_stout=1, c_sw=1.7, m0=-0.02, prec=prec, seed=71)
    b = np.stack([synth.gaussian_spinor(s.V, 72 + r) for r in range(n)])
    x0 = np.stack([0.1 * synth.gaussian_spinor(s.V, 90 + r) for r in range(n)])
    fb, fx0 = s.lat.to_field(b, prec), s.lat.to_field(x0, prec)
    start = s.lat.from_field(fx0, prec, n)
    want = [s.ref.sap(block, b[r], 2, 3, x0=start[r] if guess else None) for r in range(n)]
    for k in range(1 if guess else variants):
        fx = fx0.clone()
        with forced_variant(k):
            s.op.sap_smooth(fb, fx, 2, 3, nrhs=n, x_is_zero=not guess)
        got = s.lat.from_field(fx, prec, n)
        for r in range(n):
            assert relerr(got[r], want[r]) <= SAP_TOL[prec], (k, r)
    dd.device_status()   # no staging wait expired
    s.close()
