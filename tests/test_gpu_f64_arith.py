"""GPU: FP64 steps against the FP64 oracle where their own reciprocals, ratios and series
orders change: tiny and huge densities (beyond the range of the ratio, which takes the exact
recomputation), |x| on both sides of each series bound (2^-10, 2^-7, 2^-4, 2^-2), and
non-positive populations.  Kn and neq sum nine terms, each with a few roundings of the
population (u = 2^-53): |dKn| <= 18 * 9 u; KL's terms are x f^neq, so |dKL| <= 18 u sum|f^neq|
plus the truncation and rounding of the series, 2^-52 of KL."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu
U = 2.0 ** -53


def _state(nx, ny, amp, scale):
    rng = np.random.default_rng(17)
    w = np.array([4 / 9] + [1 / 9] * 4 + [1 / 36] * 4)[:, None, None]
    return w * scale * (1.0 + amp * rng.uniform(-1, 1, (9, ny, nx)))


@pytest.mark.parametrize("amp", [1e-4, 2e-3, 1e-2, 0.05, 0.2, 0.5, 1.3])
@pytest.mark.parametrize("scale", [1.0, 1e-290, 1e280])
def test_f64_sensors(amp, scale):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2603_13618_gb300 import kss

    nx, ny, tau = 97, 13, 0.9
    f = _state(nx, ny, amp, scale)
    ref, _ = oracle.sensor_fields(f, tau, pull=True)
    new = oracle.step(f, tau)
    with kss.Lattice(nx, ny, precision="fp64", tau=tau, record=("kn", "kl", "neq")) as lat:
        lat.set_populations(f)
        lat.step(1)
        got = {s: lat.read_sensor(s) for s in ("kn", "kl", "neq")}
        np.testing.assert_allclose(lat.get_populations(), new, rtol=0,
                                   atol=64 * U * np.max(np.abs(new)))
    neq = ref[oracle.SENSOR_ID["neq"]]
    for name in ("kn", "kl", "neq"):
        want = ref[oracle.SENSOR_ID[name]]
        fin = np.isfinite(want)
        np.testing.assert_array_equal(np.isinf(got[name]), ~fin)
        # (Kn's terms x have errors of u f / f^eq, at most u (1 + |x|) each)
        bound = {"kn": 18 * 9 * U * (1 + np.abs(want)), "neq": 18 * U * 2 * scale * (1 + amp),
                 "kl": 18 * U * (neq + scale * 1e-300) * (1 + amp) + 8 * U * np.abs(want)}[name]
        err = np.abs(got[name] - want)
        assert np.all(err[fin] <= np.broadcast_to(bound, err.shape)[fin]), (
            name, float(np.nanmax((err / bound)[fin])))
