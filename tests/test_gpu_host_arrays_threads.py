"""GPU: more threads in calls at once than there are page-locked buffers to borrow; the calls
that find none copy through the driver, with the same results."""
import threading

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_more_threads_than_buffers():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2603_13618_gb300 import inputs, kss

    nthreads, rounds = 24, 12
    start = threading.Barrier(nthreads)
    results, failed = {}, []

    def work(k, alone):
        try:
            nx, ny = 40 + 3 * (k % 5), 50 - (k % 5)
            with kss.Lattice(nx, ny, stream="own") as lat:
                if not alone:
                    start.wait(timeout=60)
                got = []
                for r in range(rounds):
                    lat.set_fields(*inputs.random_smooth(nx, ny, seed=100 * (k % 5) + r, kmax=2))
                    lat.step(2)
                    got += [*lat.read_moments(), lat.read_sensor("kl"), *lat.read_flags(),
                            lat.read_stats()[0], lat.get_populations()]
                    boxes, mask = lat.regrid()
                    got += [np.array(boxes), mask]
                results[k, alone] = got
        except Exception as e:  # reported by the main thread
            failed.append(e)
            start.abort()

    threads = [threading.Thread(target=work, args=(k, False)) for k in range(nthreads)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for k in range(5):
        work(k, True)
    assert not failed, failed
    for k in range(nthreads):
        for a, b in zip(results[k, False], results[k % 5, True]):
            np.testing.assert_array_equal(a, b)
