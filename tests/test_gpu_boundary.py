"""GPU: the copies between pitched planes and dense FP64 arrays (populations, sensor fields)
are exact conversions, whatever the width and the alignment of the dense array: FP32 values
come back as themselves (NaN as NaN), FP64 inputs rounded to nearest even as numpy rounds."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch_cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    return torch


def _values(shape):
    """FP64 values over the FP32 range: ordinary, at rounding boundaries, subnormal, zero,
    huge, infinite and NaN."""
    rng = np.random.default_rng(5)
    v = rng.standard_normal(shape) * 2.0 ** rng.integers(-40, 40, shape)
    tie = np.float32(rng.standard_normal(shape)).astype(np.float64)
    v = np.where(rng.random(shape) < 0.3, tie + np.spacing(np.float32(tie)) / 2.0, v)
    odd = np.array([0.0, -0.0, 1e-40, -1e-45, 3.5e38, np.inf, -np.inf, np.nan, 1.1754943e-38])
    return np.where(rng.random(shape) < 0.1, rng.choice(odd, shape), v)


@pytest.mark.parametrize("offset", [0, 1])
@pytest.mark.parametrize("nx,ny", [(1, 3), (2, 1), (129, 5), (516, 3), (1030, 2)])
def test_population_copies_are_exact(torch_cuda, nx, ny, offset):
    torch = torch_cuda
    from paper_2603_13618_gb300 import kss

    f = _values((9, ny, nx))
    buf = torch.zeros(f.size + offset, dtype=torch.float64, device="cuda")
    buf[offset:] = torch.from_numpy(f.reshape(-1))
    dev = buf[offset:].view(9, ny, nx)  # offset 1: 8-byte aligned only
    with np.errstate(over="ignore"):
        want = f.astype(np.float32).astype(np.float64)
    with kss.Lattice(nx, ny, precision="fp32", output_every=0) as lat:
        for src in (dev, f):
            lat.set_populations(src)
            np.testing.assert_array_equal(lat.get_populations(), want)
            np.testing.assert_array_equal(lat.get_populations(device=True).cpu().numpy(), want)


@pytest.mark.parametrize("offset", [0, 1])
@pytest.mark.parametrize("nx,ny", [(1, 3), (130, 5), (517, 9)])
def test_sensor_copies_do_not_depend_on_alignment(torch_cuda, nx, ny, offset):
    torch = torch_cuda
    from paper_2603_13618_gb300 import inputs, kss

    with kss.Lattice(nx, ny, precision="fp32", record=("kl",)) as lat:
        lat.set_fields(*inputs.random_smooth(nx, ny, seed=3, kmax=2))
        lat.step(3)
        want = lat.read_sensor("kl")
        buf = torch.zeros(nx * ny + offset, dtype=torch.float64, device="cuda")
        out = buf[offset:].view(ny, nx)
        lat.read_sensor("kl", out=out)
        np.testing.assert_array_equal(out.cpu().numpy(), want)
        np.testing.assert_array_equal(want, want.astype(np.float32))
