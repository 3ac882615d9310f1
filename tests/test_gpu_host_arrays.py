"""GPU: small host arrays travel through page-locked memory that calls borrow from a pool.
What arrives is what device arrays hold, on both sides of the size line (1 MiB less the
256-byte status block), and with several threads on lattices of their own at once."""
import threading

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


def _same(lat, steps):
    lat.step(steps)
    for name in ("kl", "neq"):
        np.testing.assert_array_equal(lat.read_sensor(name),
                                      lat.read_sensor(name, device=True).cpu().numpy())
    for a, b in zip(lat.read_moments(), lat.read_moments(device=True)):
        np.testing.assert_array_equal(a, b.cpu().numpy())
    (f, t, c), (g, u, d) = lat.read_flags(), lat.read_flags(device=True)
    np.testing.assert_array_equal(f, g.cpu().numpy())
    np.testing.assert_array_equal(t, u.cpu().numpy())
    np.testing.assert_array_equal(c, d)
    np.testing.assert_array_equal(c[:2], [(f & 1).sum(), ((f >> 1) & 1).sum()])
    np.testing.assert_array_equal(lat.get_populations(),
                                  lat.get_populations(device=True).cpu().numpy())


# (one field of FP64, and three, just below and above 1 048 320 bytes; nine planes of them)
@pytest.mark.parametrize("nx,ny", [(1, 1), (120, 121), (121, 121), (208, 210), (209, 209),
                                   (361, 363), (362, 362)])
def test_host_arrays_equal_device_arrays(kss, nx, ny):
    import torch

    from paper_2603_13618_gb300 import inputs

    f = inputs.random_smooth(nx, ny, seed=4, kmax=3)
    with kss.Lattice(nx, ny) as a, kss.Lattice(nx, ny) as b:
        for fields in (f, [x.astype(np.float32) for x in f]):
            a.set_fields(*fields)
            b.set_fields(*(torch.from_numpy(x).cuda() for x in fields))
            np.testing.assert_array_equal(a.get_populations(), b.get_populations())
        p = a.get_populations()
        a.set_populations(p)
        np.testing.assert_array_equal(a.get_populations(), p)
        _same(a, 2)


def test_threads_do_not_share_what_they_borrow(kss):
    from paper_2603_13618_gb300 import inputs

    failed = []

    def work(k):
        try:
            nx, ny = 60 + 7 * k, 90 - 5 * k
            with kss.Lattice(nx, ny, stream="own") as lat:
                for r in range(8):
                    lat.set_fields(*inputs.random_smooth(nx, ny, seed=10 * k + r, kmax=2))
                    sums = lat.read_stats()[0]
                    rho = lat.read_moments()[0]
                    np.testing.assert_allclose(sums[0], rho.sum(), rtol=1e-6)
                    lat.step(3)
                    kl = lat.read_sensor("kl")
                    flags, _, counts = lat.read_flags()
                    assert (flags & 1).sum() == counts[0]
                    np.testing.assert_array_equal(kl, lat.read_sensor("kl"))
        except Exception as e:  # reported by the main thread
            failed.append(e)

    threads = [threading.Thread(target=work, args=(k,)) for k in range(8)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failed, failed
