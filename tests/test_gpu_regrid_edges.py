"""GPU: regridding against the oracle (integer work, compared exactly) where its kernels
change path: tile grids whose box signatures exceed a warp's shared memory (512 values),
buffers wider than a tile and than the lattice, rows that are not 8-byte aligned, and device
outputs that are 4-byte aligned only."""
import ctypes

import numpy as np
import pytest

from oracle import regrid as orc_regrid

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch_cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    return torch


def _flags(ny, nx, seed, cells):
    rng = np.random.default_rng(seed)
    f = np.zeros((ny, nx), dtype=np.uint8)
    for _ in range(cells):
        y, x = rng.integers(0, ny), rng.integers(0, nx)
        f[y:y + rng.integers(1, 1 + max(1, ny // 5)), x:x + rng.integers(1, 1 + max(1, nx // 5))] |= 1
    f[rng.random((ny, nx)) < 0.3] |= 2
    return f


@pytest.mark.parametrize("ny,nx,tile,buf,eff,cells", [
    (2200, 2300, 8, 2, 0.9, 6), (8, 4120, 8, 2, 0.9, 9), (70, 90, 8, 11, 0.8, 2),
    (40, 33, 8, 100, 0.9, 1), (129, 257, 16, 17, 0.98, 3), (64, 72, 8, 1, 0.98, 9),
    (300, 1001, 8, 0, 0.95, 20)])
def test_regrid_edges(torch_cuda, ny, nx, tile, buf, eff, cells):
    torch = torch_cuda
    from paper_2603_13618_gb300 import kss

    flags = _flags(ny, nx, ny + nx, cells)
    want_mask = orc_regrid.tile_mask(flags, tile, buf)
    want = orc_regrid.cluster(want_mask, eff)
    got, mask = kss.regrid_flags(flags, tile=tile, buffer=buf, efficiency=eff)
    np.testing.assert_array_equal(mask, want_mask)
    assert got == want

    # device arrays: flags one byte off any alignment, boxes four bytes off
    dev = torch.zeros(flags.size + 1, dtype=torch.uint8, device="cuda")
    dev[1:] = torch.from_numpy(flags.reshape(-1))
    n = max(1, len(want))
    boxes = torch.full((4 * n + 1,), -7, dtype=torch.int32, device="cuda")
    dmask = torch.zeros(want_mask.size, dtype=torch.uint8, device="cuda")
    count = ctypes.c_int32()
    rc = kss.load().kss_regrid_flags(
        ctypes.c_void_p(dev.data_ptr() + 1), nx, ny, tile, buf, eff,
        ctypes.c_void_p(dmask.data_ptr()),
        ctypes.cast(ctypes.c_void_p(boxes.data_ptr() + 4), ctypes.c_void_p), n,
        ctypes.byref(count), 1, torch.cuda.current_stream().cuda_stream)
    assert rc == 0 and count.value == len(want)
    np.testing.assert_array_equal(dmask.cpu().numpy().reshape(want_mask.shape), want_mask)
    out = boxes.cpu().numpy()
    assert out[0] == -7
    assert [tuple(b) for b in out[1:].reshape(-1, 4)[:len(want)].tolist()] == want
