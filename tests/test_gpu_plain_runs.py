"""GPU: runs of plain FP32 steps, which go two to a launch, against the same steps one call
each: populations, and the outputs of the output steps among them, bit for bit, at widths
around a tile's 128 columns and a lane's four and heights around its eight rows."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def kss():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2603_13618_gb300 import kss

    return kss


@pytest.mark.parametrize("every", [1000, 4])
@pytest.mark.parametrize("nx,ny", [(1, 1), (3, 2), (5, 40), (127, 8), (128, 9), (129, 16), (130, 7),
                                   (256, 33), (381, 65), (1021, 517)])
def test_runs_equal_single_steps(kss, nx, ny, every):
    from paper_2603_13618_gb300 import inputs

    fields = inputs.smooth_jump(nx, ny, seed=3, kmax=2)
    kw = dict(precision="fp32", tau=0.57, record=("kl",), output_every=every)
    with kss.Lattice(nx, ny, **kw) as a, kss.Lattice(nx, ny, **kw) as b:
        for x in (a, b):
            x.set_fields(*fields)
        for n in (2, 3, 7, 7, 2, 3, 8):
            a.step(n)
            for _ in range(n):
                b.step(1)
            np.testing.assert_array_equal(a.get_populations(), b.get_populations())
            if every == 4:
                np.testing.assert_array_equal(a.read_sensor("kl"), b.read_sensor("kl"))
                np.testing.assert_array_equal(a.read_sensor("s"), b.read_sensor("s"))
                np.testing.assert_array_equal(a.read_flags()[0], b.read_flags()[0])
