"""GPU: an all-sensor step evaluates only the sensors that it records or tags.  Whatever the
subset, each field, the flags, the tile counts and the sums are those of a step that records
all of Table 1, bit for bit (the same arithmetic per sensor), at widths around the 32-column
passes of a warp and around a ragged row end."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SUBSETS = [("s",), ("qh", "tau_ns"), ("hr",), ("sigma_h",), ("sigma_kl",), ("alpha",),
           ("c", "neq"), ("hr", "kl"), ("alpha", "kn"), ("e", "sigma_kl", "qe")]


@pytest.mark.parametrize("precision", ["fp32", "fp64", "fp16dev"])
@pytest.mark.parametrize("nx,ny,tau2", [(1, 3, 0.0), (33, 17, 1.4), (129, 40, 0.0), (254, 9, 1.1)])
def test_subsets_equal_the_whole_table(precision, nx, ny, tau2):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2603_13618_gb300 import inputs, kss

    fields = inputs.smooth_jump(nx, ny, seed=21, kmax=2)
    flag = dict(refine_sensor="s", refine_threshold=2e-3, switch_sensor="e",
                switch_threshold=1e-3)

    def run(record):
        with kss.Lattice(nx, ny, precision=precision, tau=0.7, tau2=tau2, record=record,
                         **flag) as lat:
            lat.set_fields(*fields)
            lat.step(3)
            out = {s: lat.read_sensor(s) for s in record}
            return out, lat.read_flags(), lat.read_stats(), lat.get_populations()

    whole, flags, stats, pops = run(kss.SENSORS)
    for subset in SUBSETS:
        got, f, st, p = run(subset)
        for s in subset:
            np.testing.assert_array_equal(got[s], whole[s], err_msg=f"{subset} {s}")
        for a, b in zip((*f, *st, p), (*flags, *stats, pops)):
            np.testing.assert_array_equal(a, b, err_msg=str(subset))
