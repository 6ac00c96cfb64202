"""The residual b - D x of a Schwarz phase sees x as it is stored, in FP32, and
the links of the block solves (16-bit storage): in the first sweep from a given
x, and in every phase of the two-level preconditioner's smoother.

The FP64 oracle works on the very fields of the kernels: c_sw = 0 and m0 = 0 (A
= 4, A^-1 = 1/4), and links that 16 bits hold exactly (colour permutations
times powers of i) or the nine entries as rounded to the storage. The only
roundings left are those of the iterate and of FP32 arithmetic."""
import numpy as np
import pytest

import oracle
import paper_1710_07041_gb300 as dd
import synth

pytestmark = pytest.mark.gpu

CASES = [((8, 8, 8, 8), (4, 4, 4, 4)), ((16, 8, 8, 8), (8, 4, 4, 4)), ((8, 4, 8, 8), (4, 2, 4, 4))]
# unit in the last place of the storage, relative to the power of two below a value
ULP = {dd.F16: 2.0 ** -10, dd.BF16: 2.0 ** -7}


def exact_links(V, seed):
    """Links that every storage holds exactly: permutations of the colours
    (even ones) times diag(i^a, i^b, i^c) of determinant 1."""
    rng = np.random.default_rng(seed)
    U = np.zeros((V * 4, 3, 3), dtype=np.complex128)
    a, b, k = (rng.integers(0, n, V * 4) for n in (4, 4, 3))
    for row, ph in enumerate((a, b, -(a + b))):
        U[np.arange(V * 4), row, (row + k) % 3] = np.array([1, 1j, -1, -1j])[ph % 4]
    return U.reshape(V, 4, 3, 3)


def rounded(z, prec):
    """Every component rounded to the storage, to nearest even."""
    v = parts(z)
    if prec == dd.BF16:
        m, e = np.frexp(v)
        v = np.ldexp(np.rint(np.ldexp(m, 8)), e - 8)
    else:
        v = v.astype(np.float16).astype(np.float64)
    return np.ascontiguousarray(v).view(np.complex128)


def colour_mask(ref, block, colour):
    """Sites of the blocks of one colour."""
    on = np.zeros(ref.V, dtype=bool)
    for k in range(ref.nblocks(block)):
        if ref.block_colour(block, k) == colour:
            on[ref.block_sites(block, k)] = True
    return on


def phase(ref, block, colour, b, x, nmr):
    """The colour's corrections to x: the block solves of b - D x."""
    r, e = b - ref.apply(x), np.zeros_like(x)
    for k in range(ref.nblocks(block)):
        if ref.block_colour(block, k) == colour:
            e += ref.block_solve(block, k, r, nmr)
    return e


def parts(z):
    return np.ascontiguousarray(z).view(np.float64)


@pytest.mark.parametrize("prec", [dd.F16, dd.BF16, dd.F16N])
@pytest.mark.parametrize("dims,block", CASES)
@pytest.mark.parametrize("links", ["exact", "rounded"])
def test_second_colour_sees_the_stored_iterate(prec, dims, block, links):
    """One sweep from a given x. The blocks of the first colour are final after
    their phase, so the x that the second colour works on is known as stored,
    and its result is round(x + e). Bound, each component: half a unit in the
    last place of the storage plus 2^-17 (128 FP32 roundoffs) of the largest
    component for the arithmetic."""
    V = int(np.prod(dims))
    U = exact_links(V, 5) if links == "exact" else synth.gauge(dims, 0.3, 1, 0.1, 5)
    lat = dd.Lattice(dims, block)
    gauge = dd.Gauge(lat, U)
    op = dd.Op(gauge, 0.0, 0.0, prec)
    ref = oracle.Operator(dims, U if links == "exact" else rounded(U, prec), 0.0, 0.0)
    fb, fx = lat.to_field(synth.gaussian_spinor(V, 6), prec), lat.to_field(synth.gaussian_spinor(V, 7), prec)
    b, x = lat.from_field(fb, prec), lat.from_field(fx, prec)
    op.sap_smooth(fb, fx, 1, 4, x_is_zero=False)
    got = lat.from_field(fx, prec)
    second = colour_mask(ref, block, 1)
    x[~second] = got[~second]
    want = parts((x + phase(ref, block, 1, b, x, 4))[second])
    if prec == dd.F16N:   # fixed point, a step of the site's largest component / 32767
        step = np.repeat(np.abs(want.reshape(-1, 24)).max(axis=1), 24).reshape(want.shape) / 32767
    else:
        step = ULP[prec] * 2.0 ** np.floor(np.log2(np.abs(want)))
    off = np.abs(parts(got[second]) - want) - 0.5 * step - 2.0 ** -17 * np.abs(want).max()
    assert off.max() <= 0, (int((off > 0).sum()), off.size)
    op.close()
    gauge.close()
    lat.close()


@pytest.mark.parametrize("prec", [dd.F16, dd.BF16])
@pytest.mark.parametrize("dims,block", [((8, 8, 8, 8), (4, 4, 4, 4)), ((8, 4, 8, 8), (4, 2, 4, 4))])
def test_two_level_smoother_works_on_the_stored_iterate(prec, dims, block):
    """Test vectors on two colours and a residual on the third: the coarse part
    vanishes, so the preconditioner's result is the smoother's x, whose phases
    are followed one by one, x rounded to the storage after each. FP32 noise
    of 8 roundoffs (2^-21) crosses a rounding boundary in one of ULP / 2^-19
    components, an error of sqrt(2^-19 / ULP) ULP <= ULP / 22 in the 2-norm;
    bound ULP / 16. (Residuals or corrections handed on in 16 bits: each a
    rounding of 0.2 to 0.3 ULP.)"""
    V = int(np.prod(dims))
    U = exact_links(V, 8)
    lat = dd.Lattice(dims, block)
    gauge = dd.Gauge(lat, U)
    op = dd.Op(gauge, 0.0, 0.0, prec)
    ref = oracle.Operator(dims, U, 0.0, 0.0)
    tv = np.stack([synth.gaussian_spinor(V, 20 + k) for k in range(4)])
    tv[..., 2] = 0
    mg = dd.Multigrid(op, tv, setup_iters=0, sweeps=2, mr_steps=4)
    r = synth.gaussian_spinor(V, 9)
    r[..., :2] = 0
    r = lat.from_field(lat.to_field(r, prec), prec)
    rf, xf = lat.to_field(r, dd.F32), lat.new_field(dd.F32)
    mg.precondition(rf, xf)
    got = lat.from_field(xf, dd.F32)
    x = np.zeros_like(r)
    for _ in range(2):
        for colour in range(2):
            x = rounded(x + phase(ref, block, colour, r, x, 4), prec)
    err = np.linalg.norm(got - x) / np.linalg.norm(x)
    print(f"two-level smoother error {err / ULP[prec]:.4f} ULP")
    assert err <= ULP[prec] / 16
    mg.close()
    op.close()
    gauge.close()
    lat.close()
