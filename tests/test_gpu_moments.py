"""GPU: kss_read_moments against FP64 arithmetic on the same populations.

FP32 populations whose sums are exact in FP64 take an integer path: its density is the FP64
sum bit for bit, and its velocities the rounded quotient (the corrected quotient is within
2^-86 of the exact one before it is rounded, so it could differ from IEEE division only
within 2^-33 of a rounding boundary).  Every other cell is FP64 arithmetic itself.  So the
results are compared for equality.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

W = np.array([4 / 9] + [1 / 9] * 4 + [1 / 36] * 4)[:, None, None]


def _populations(kind, ny, nx):
    rng = np.random.default_rng(11)
    f = W * (1.0 + 0.1 * rng.standard_normal((9, ny, nx)))
    if kind == "rest":  # exact rest states and single-velocity cells
        f = W * 2.0 ** rng.integers(-3, 4, (1, ny, nx))
    elif kind == "span":  # exponents 24, 25 and 26 apart: both sides of the integer path
        f[rng.integers(0, 9, ny * nx), np.repeat(np.arange(ny), nx), np.tile(np.arange(nx), ny)] \
            *= 2.0 ** -rng.integers(20, 24, ny * nx)
    elif kind == "signed":  # non-positive and zero populations
        f = np.where(rng.random(f.shape) < 0.02, -f, np.where(rng.random(f.shape) < 0.02, 0, f))
    elif kind == "edge":  # subnormal, huge and infinite populations
        f = f * 2.0 ** rng.choice([-130, -126, 0, 120], (1, ny, nx))
        f[rng.random(f.shape) < 0.01] = np.inf
    return f.astype(np.float32).astype(np.float64)


def _moments(v):
    with np.errstate(all="ignore"):
        r = ((v[0] + v[1]) + (v[2] + v[3])) + ((v[4] + v[5]) + (v[6] + v[7])) + v[8]
        jx = (v[1] + v[5] + v[8]) - (v[3] + v[6] + v[7])
        jy = (v[2] + v[5] + v[6]) - (v[4] + v[7] + v[8])
        return r, jx / r, jy / r


@pytest.mark.parametrize("precision", ["fp32", "fp16dev"])
@pytest.mark.parametrize("kind", ["near", "rest", "span", "signed", "edge"])
@pytest.mark.parametrize("nx,ny", [(1, 1), (257, 33), (512, 7)])
def test_moments_are_those_of_fp64_arithmetic(precision, kind, nx, ny):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2603_13618_gb300 import kss

    with kss.Lattice(nx, ny, precision=precision, output_every=0) as lat:
        lat.set_populations(_populations(kind, ny, nx))
        want = _moments(lat.get_populations())
        for got, ref in zip(lat.read_moments(), want):
            np.testing.assert_array_equal(got, ref)
