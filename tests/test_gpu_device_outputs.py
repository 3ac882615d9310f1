"""GPU: flags, tile counts, tile masks and boxes written to device memory at any byte offset:
the kernels' 16-, 4- and 1-byte paths, and the driver's copy for elements off their boundary.
The bytes before and after stay as they were."""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

MARK = 0xA5


@pytest.fixture(scope="module")
def kss():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2603_13618_gb300 import kss

    return kss


class Room:
    """Device bytes around an output `offset` bytes into an allocation (256-byte aligned)."""

    def __init__(self, nbytes, offset):
        import torch

        self.raw = torch.full((nbytes + offset + 64,), MARK, dtype=torch.uint8, device="cuda")
        assert self.raw.data_ptr() % 256 == 0
        self.nbytes, self.offset = nbytes, offset
        self.ptr = ctypes.c_void_p(self.raw.data_ptr() + offset)

    def bytes(self, written=None):
        written = self.nbytes if written is None else written
        a = self.raw.cpu().numpy()
        assert (a[:self.offset] == MARK).all() and (a[self.offset + written:] == MARK).all()
        return a[self.offset:self.offset + written].tobytes()


@pytest.mark.parametrize("nx,ny", [(64, 5), (68, 7), (33, 40), (304, 66)])
@pytest.mark.parametrize("flags_at,tiles_at", [(0, 0), (16, 4), (8, 8), (4, 1), (2, 2), (1, 3)])
def test_flags_and_tile_counts(kss, nx, ny, flags_at, tiles_at):
    from paper_2603_13618_gb300 import inputs

    with kss.Lattice(nx, ny, precision="fp32", tau=0.6, tile=8) as lat:
        lat.set_fields(*inputs.smooth_jump(nx, ny, seed=4, kmax=3))
        lat.step(2)
        flags, tiles, counts = lat.read_flags()
        assert 0 < counts[0]
        f, t = Room(flags.nbytes, flags_at), Room(tiles.nbytes, tiles_at)
        c = (ctypes.c_int64 * 3)()
        lat._check(lat._lib.kss_read_flags(lat._h, f.ptr, t.ptr, c, 1))
        assert f.bytes() == flags.tobytes() and t.bytes() == tiles.tobytes()
        assert list(c) == list(counts)
        f, t = Room(flags.nbytes, flags_at), Room(tiles.nbytes, tiles_at)
        lat._check(lat._lib.kss_read_flags(lat._h, f.ptr, None, None, 1))
        lat._check(lat._lib.kss_read_flags(lat._h, None, t.ptr, None, 1))
        assert f.bytes() == flags.tobytes() and t.bytes() == tiles.tobytes()


@pytest.mark.parametrize("mask_at,boxes_at", [(0, 0), (1, 4), (3, 8), (0, 1), (5, 2)])
def test_tile_mask_and_boxes(kss, mask_at, boxes_at):
    import torch

    from paper_2603_13618_gb300 import inputs

    nx, ny = 200, 130
    fields = inputs.smooth_jump(nx, ny, seed=4, kmax=3)
    with kss.Lattice(nx, ny, precision="fp32", tau=0.6, tile=8) as lat:
        lat.set_fields(*fields)
        lat.step(2)
        tenth = float(np.quantile(lat.read_sensor("kn"), 0.9))  # tag a tenth of the cells
    with kss.Lattice(nx, ny, precision="fp32", tau=0.6, tile=8, refine_threshold=tenth) as lat:
        lat.set_fields(*fields)
        lat.step(2)
        boxes, mask = lat.regrid()
        assert len(boxes) > 1
        want = np.array(boxes, dtype=np.int32)
        flags = lat.read_flags(device=True)[0]
        n = ctypes.c_int32()
        stream = torch.cuda.current_stream().cuda_stream
        for room in (len(boxes) + 3, len(boxes) - 1):  # boxes beyond the caller's room are left out
            written = min(room, len(boxes)) * 16
            m, b = Room(mask.nbytes, mask_at), Room(room * 16, boxes_at)
            lat._check(lat._lib.kss_regrid(lat._h, 2, 0.98, m.ptr, b.ptr, room, ctypes.byref(n), 1))
            assert n.value == len(boxes) and m.bytes() == mask.tobytes()
            assert b.bytes(written) == want.tobytes()[:written]
            m, b = Room(mask.nbytes, mask_at), Room(room * 16, boxes_at)
            lat._check(lat._lib.kss_regrid_flags(ctypes.c_void_p(flags.data_ptr()), nx, ny, 8, 2,
                                                 0.98, m.ptr, b.ptr, room, ctypes.byref(n), 1,
                                                 stream))
            assert n.value == len(boxes) and m.bytes() == mask.tobytes()
            assert b.bytes(written) == want.tobytes()[:written]
