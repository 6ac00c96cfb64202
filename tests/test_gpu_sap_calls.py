"""Forms of the smoother call on the packed kernel's blocks, bit for bit against
single calls: several lattices at once from a given x (a residual of each), more
right-hand sides than one launch takes, and calls inside a stream capture of the
caller's, as the first ones of a process and after others."""
import os
import subprocess
import sys

import numpy as np
import pytest
import torch

import paper_1710_07041_gb300 as dd
import synth
from gpu_common import Setup

pytestmark = pytest.mark.gpu

BLOCKS = [((8, 8, 8, 8), (8, 8, 8, 16), (4, 4, 4, 4)), ((16, 8, 8, 8), (16, 8, 16, 8), (8, 4, 4, 4))]
SETUP = dict(eps=0.3, n_stout=1, c_sw=1.7, m0=-0.02)


def fields(s, prec, n, seed):
    b = np.stack([synth.gaussian_spinor(s.V, seed + r) for r in range(n)])
    x = np.stack([0.1 * synth.gaussian_spinor(s.V, seed + 100 + r) for r in range(n)])
    return s.lat.to_field(b, prec), s.lat.to_field(x, prec)


@pytest.mark.parametrize("prec", [dd.F32, dd.F16, dd.BF16, dd.F16N])
@pytest.mark.parametrize("small,large,block", BLOCKS)
@pytest.mark.parametrize("guess", [False, True])
def test_several_lattices(prec, small, large, block, guess):
    ss = [Setup(d, block, prec=prec, seed=80 + i, **SETUP) for i, d in enumerate((small, large, small))]
    n = (2, 1, 3)
    f = [fields(s, prec, k, 200 * (i + 1)) for i, (s, k) in enumerate(zip(ss, n))]
    alone = [x.clone() for _, x in f]
    for s, k, (b, _), x in zip(ss, n, f, alone):
        s.op.sap_smooth(b, x, 2, 3, nrhs=k, x_is_zero=not guess)
    dd.sap_smooth_multi([(s.op, b, x, k) for s, k, (b, x) in zip(ss, n, f)], 2, 3, x_is_zero=not guess)
    for x, (_, y) in zip(alone, f):
        assert torch.equal(x, y)
    for s in ss:
        s.close()


@pytest.mark.parametrize("prec", [dd.F32, dd.BF16])
@pytest.mark.parametrize("dims,block", [b[::2] for b in BLOCKS])
def test_more_right_hand_sides_than_a_launch_takes(prec, dims, block):
    s = Setup(dims, block, prec=prec, seed=83, **SETUP)
    n = 67
    b, x = fields(s, prec, 3, 300)
    size = b.numel() // 3
    pick = [r % 3 for r in range(n)]
    bn, xn = (torch.cat([f[size * r:size * (r + 1)] for r in pick]) for f in (b, x))
    s.op.sap_smooth(bn, xn, 2, 3, nrhs=n, x_is_zero=False)
    s.op.sap_smooth(b, x, 2, 3, nrhs=3, x_is_zero=False)
    for k, r in enumerate(pick):
        assert torch.equal(xn[size * k:size * (k + 1)], x[size * r:size * (r + 1)]), k
    s.close()


def captured(prec, dims, block, guess):
    """The smoother in a capture of the caller's, replayed twice on the given x."""
    s = Setup(dims, block, prec=prec, seed=84, **SETUP)
    b, x0 = fields(s, prec, 2, 400)
    x = x0.clone()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        s.op.sap_smooth(b, x, 2, 3, nrhs=2, x_is_zero=not guess)
    out = []
    for _ in range(2):
        x.copy_(x0)
        g.replay()
        out.append(s.lat.from_field(x, prec, 2))
    return s, b, x0, out


CHILD = """
import sys
import numpy as np
import torch
from test_gpu_sap_calls import captured
a = eval(sys.argv[1])
s, b, x0, out = captured(*a)
x = x0.clone()
s.op.sap_smooth(b, x, 2, 3, nrhs=2, x_is_zero=not a[3])
assert (out[0] == out[1]).all() and (out[0] == s.lat.from_field(x, a[0], 2)).all()
"""


@pytest.mark.parametrize("prec", [dd.F32, dd.F16])
@pytest.mark.parametrize("dims,block", [b[::2] for b in BLOCKS])
@pytest.mark.parametrize("guess", [False, True])
def test_inside_a_capture(prec, dims, block, guess):
    s, b, x0, out = captured(prec, dims, block, guess)
    x = x0.clone()
    s.op.sap_smooth(b, x, 2, 3, nrhs=2, x_is_zero=not guess)
    assert (out[0] == out[1]).all() and (out[0] == s.lat.from_field(x, prec, 2)).all()
    s.close()


@pytest.mark.parametrize("case", [(dd.F32, (8, 8, 8, 8), (4, 4, 4, 4), True),
                                  (dd.F16, (16, 8, 8, 8), (8, 4, 4, 4), False)])
def test_first_call_of_a_process_inside_a_capture(case):
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    env = dict(os.environ, PYTHONPATH=os.pathsep.join([root, os.path.join(root, "tests")]))
    p = subprocess.run([sys.executable, "-c", CHILD, repr(case)], cwd=root, env=env, capture_output=True, text=True,
                       timeout=600)
    assert p.returncode == 0, p.stdout[-2000:] + p.stderr[-4000:]
