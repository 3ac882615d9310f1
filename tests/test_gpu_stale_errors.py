"""GPU: an error that the caller's own CUDA calls left behind (one that does not lose the
context) is not taken for a failure of the calls that wait and read flags, counts and sums."""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _runtime():
    """The CUDA runtime library that this process uses."""
    with open("/proc/self/maps") as fh:
        paths = {line.split()[-1] for line in fh if "libcudart.so" in line}
    assert len(paths) == 1, paths
    return ctypes.CDLL(paths.pop())


@pytest.mark.parametrize("call", ["sync", "read_stats", "read_flags", "read_flags_device"])
def test_a_stale_error_is_not_ours(call):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2603_13618_gb300 import inputs, kss

    with kss.Lattice(70, 45, precision="fp32", tau=0.7) as lat:
        lat.set_fields(*inputs.smooth_jump(70, 45, seed=3, kmax=3))
        lat.step(3)
        lat.sync()
        want = lat.read_flags()
        out = None
        if call == "read_flags_device":
            out = tuple(torch.empty(x.shape, dtype=torch.from_numpy(x).dtype, device="cuda")
                        for x in want[:2])
        rt = _runtime()
        assert rt.cudaSetDevice(100000) != 0 and rt.cudaPeekAtLastError() != 0
        try:
            if call == "sync":
                lat.sync()
            elif call == "read_stats":
                np.testing.assert_array_equal(lat.read_stats()[1], want[2])
            else:
                got = lat.read_flags(out=out)
                rt.cudaGetLastError()
                for a, b in zip(got, want):
                    np.testing.assert_array_equal(a.cpu().numpy() if hasattr(a, "cpu") else a, b)
        finally:
            rt.cudaGetLastError()
