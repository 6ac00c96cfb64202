"""Rounding errors of the packed Schwarz kernel in FP32 storage against those
of the general kernel, which recomputes the even sites' correction from the odd
ones'. The relative L2 error of 98304 components spreads by 0.3% from input to
input; bound: the general kernel's, mean of four inputs, times 1.03."""
import os
import subprocess
import sys

import numpy as np
import pytest

import paper_1710_07041_gb300 as dd
import synth
from gpu_common import Setup, relerr

pytestmark = pytest.mark.gpu

DIMS, STEPS, SEEDS = (16, 8, 8, 8), (2, 4, 6), (61, 62, 63, 64)


def smoothed(block, guess):
    """One sweep, for every number of MR steps and every input."""
    out = []
    s = Setup(DIMS, block, eps=0.25, n_stout=2, c_sw=1.7, m0=-0.02, prec=dd.F32, seed=60)
    for nmr in STEPS:
        for seed in SEEDS:
            fb = s.lat.to_field(synth.gaussian_spinor(s.V, seed), dd.F32)
            fx = s.lat.to_field(0.1 * synth.gaussian_spinor(s.V, seed + 10), dd.F32)
            s.op.sap_smooth(fb, fx, 1, nmr, x_is_zero=not guess)
            out.append(s.lat.from_field(fx, dd.F32))
    ref = s.ref
    s.close()
    return np.stack(out).reshape(len(STEPS), len(SEEDS), *out[0].shape), ref


CHILD = """
import sys
import numpy as np
from test_gpu_sap_precision import smoothed
np.save(sys.argv[3], smoothed(tuple(map(int, sys.argv[1].split(","))), bool(int(sys.argv[2])))[0])
"""


@pytest.mark.parametrize("block", [(4, 4, 4, 4), (8, 4, 4, 4)])
@pytest.mark.parametrize("guess", [False, True])
def test_fp32_error_is_no_larger_than_the_general_kernels(block, guess, tmp_path):
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    env = dict(os.environ, DD_SAP_INCR="0",
               PYTHONPATH=os.pathsep.join([root, os.path.join(root, "tests"), os.environ.get("PYTHONPATH", "")]))
    f = str(tmp_path / "general.npy")
    p = subprocess.run([sys.executable, "-c", CHILD, ",".join(map(str, block)), str(int(guess)), f], cwd=root, env=env,
                       capture_output=True, text=True, timeout=600)
    assert p.returncode == 0, p.stdout[-2000:] + p.stderr[-4000:]
    general = np.load(f)
    packed, ref = smoothed(block, guess)
    for k, nmr in enumerate(STEPS):
        e = np.zeros((2, len(SEEDS)))
        for i, seed in enumerate(SEEDS):
            x0 = 0.1 * synth.gaussian_spinor(ref.V, seed + 10) if guess else None
            want = ref.sap(block, synth.gaussian_spinor(ref.V, seed), 1, nmr, x0=x0)
            e[:, i] = relerr(packed[k, i], want), relerr(general[k, i], want)
        e = e.mean(axis=1)
        print(f"{nmr} MR steps: packed {e[0]:.4g}, general {e[1]:.4g}")
        assert e[0] <= 1.03 * e[1], nmr


@pytest.mark.parametrize("dims,block", [((8, 8, 8, 8), (4, 4, 4, 4)), ((16, 8, 8, 8), (8, 4, 4, 4)),
                                        ((8, 4, 8, 8), (4, 2, 4, 4))])
def test_fp16_keeps_small_link_entries(dims, block):
    """Links exp(i eps lambda_1) with eps = 3 * 2^-24: FP16 holds their off-
    diagonal entries exactly (subnormal). Colour 1 of the smoothed x then comes
    from colour 0 of b through those entries alone, in proportion to eps. Bound:
    a few roundings of FP16 (2^-11 each; half of an entry, rounded, is off by a
    third)."""
    V, eps = int(np.prod(dims)), 3 * 2.0 ** -24
    U = np.tile(np.eye(3, dtype=np.complex128), (V, 4, 1, 1))
    U[..., 0, 0] = U[..., 1, 1] = np.cos(eps)
    U[..., 0, 1] = U[..., 1, 0] = 1j * np.sin(eps)
    s = Setup(dims, block, c_sw=0.0, m0=0.0, prec=dd.F16, U=U)
    b = 1e4 * synth.gaussian_spinor(V, 70)
    b[..., 1:] = 0
    fb, fx = s.lat.to_field(b, dd.F16), s.lat.new_field(dd.F16)
    s.op.sap_smooth(fb, fx, 2, 3)
    got, want = s.lat.from_field(fx, dd.F16), s.ref.sap(block, s.lat.from_field(fb, dd.F16), 2, 3)
    err = relerr(got[..., 1], want[..., 1])
    print(f"colour reached through the small entries: relerr {err:.3g}")
    assert err <= 3e-3
    s.close()
