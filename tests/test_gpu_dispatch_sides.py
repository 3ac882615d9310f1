"""GPU: both sides of the rules that choose a launch, each against the other by name.

Output steps go as split blocks (each block shared out to a cluster of CTAs), as one launch per
step, or as one multi-step launch, by the number of blocks against the number of SMs.  Every
test states the line it stands on, so that a later change of the rules cannot turn a comparison
into one of a kernel with itself: blocks(...) are the CTA blocks of 32 lanes x 16 bytes by
`rows` rows, and a batch with persistent CTAs (ctas_per_sm = 1) neither splits nor takes the
multi-step launch (include/kss.h, kss_batch_tuning)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

COLUMNS = {"fp32": 128, "fp64": 64, "fp16dev": 128}


@pytest.fixture(scope="module")
def kss():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2603_13618_gb300 import kss

    return kss


@pytest.fixture(scope="module")
def sms():
    torch = pytest.importorskip("torch")
    return torch.cuda.get_device_properties(0).multi_processor_count


def blocks(precision, nx, ny, rows=32):
    return -(-nx // COLUMNS[precision]) * -(-ny // rows)


def splits(precision, nblocks, rows, sms):
    """Do `nblocks` blocks of `rows` rows go as split blocks?  Their ranks of eight rows (FP32
    arithmetic: or sixteen, at two rows per warp) must fit at two CTAs per SM; of FP64, 10/7 as
    many."""
    if precision == "fp64":
        return 7 * nblocks * (rows // 8) <= 20 * sms
    if nblocks * (rows // 8) <= 2 * sms:
        return rows > 8
    return rows > 16 and nblocks * (rows // 16) <= 2 * sms


def outputs(lat, sums=True):
    flags, tiles, counts = lat.read_flags()
    out = [flags, tiles, counts, lat.get_populations(), lat.read_sensor("kl"),
           lat.read_sensor("kn")]
    return out + ([lat.read_stats()[0]] if sums else [])


def assert_equal(a, b):
    for x, y in zip(a, b):
        np.testing.assert_array_equal(x, y)


# ---- split blocks of a lone lattice against one CTA per block ----
@pytest.mark.parametrize("precision", ["fp32", "fp64", "fp16dev"])
@pytest.mark.parametrize("tile", [8, 16, 32, 64])
@pytest.mark.parametrize("nx,ny", [(1, 1), (33, 2), (128, 8), (130, 31), (257, 33), (300, 65),
                                   (600, 320)])
def test_split_lattice_against_unsplit_blocks(kss, sms, precision, tile, nx, ny):
    from paper_2603_13618_gb300 import inputs

    n = blocks(precision, nx, ny, max(32, tile))
    if (nx, ny) == (600, 320) and precision == "fp64" and tile < 64:
        assert 14 * sms < 7 * n * 4 <= 20 * sms  # (beyond the line of the other storage types)
    assert splits(precision, n, max(32, tile), sms)
    fields = inputs.smooth_jump(nx, ny, seed=5, kmax=2)
    kw = dict(precision=precision, tau=0.56, tile=tile, record=("kl",))
    batch = kss.Batch([dict(nx=nx, ny=ny)], **kw)
    batch.set_tuning(ctas_per_sm=1, multi_step=0)
    with kss.Lattice(nx, ny, **kw) as lat:
        for x in (lat, batch[0]):
            x.set_fields(*fields)
        for steps in (1, 4):
            lat.step(steps)
            batch.step(steps)
            # (a lone FP16 lattice adds its sums over 256-column blocks)
            exact = precision != "fp16dev"
            assert_equal(outputs(lat, exact), outputs(batch[0], exact))
    batch.close()


@pytest.mark.parametrize("precision,nx,ny", [("fp32", 501, 801), ("fp32", 512, 800),
                                             ("fp16dev", 1021, 805)])
def test_two_rows_per_warp_against_unsplit_blocks(kss, sms, precision, nx, ny):
    from paper_2603_13618_gb300 import inputs

    # (the FP16 lattice's blocks are 256 columns wide)
    n = blocks(precision, nx if precision == "fp32" else -(-nx // 2), ny)
    assert n * 4 > 2 * sms and splits(precision, n, 32, sms)
    fields = inputs.smooth_jump(nx, ny, seed=6, kmax=3)
    kw = dict(precision=precision, tau=0.6, record=("kl",))
    batch = kss.Batch([dict(nx=nx, ny=ny)], **kw)
    batch.set_tuning(ctas_per_sm=1, multi_step=0)
    with kss.Lattice(nx, ny, **kw) as lat:
        for x in (lat, batch[0]):
            x.set_fields(*fields)
            x.step(3) if x is lat else batch.step(3)
        exact = precision != "fp16dev"
        assert_equal(outputs(lat, exact), outputs(batch[0], exact))
    batch.close()


@pytest.mark.parametrize("nx,ny", [(33, 2), (130, 31), (300, 65), (1021, 517)])
def test_sums_of_split_fp16_blocks(kss, nx, ny):
    """The sums of the eight-cell split blocks against the four-cell unsplit ones': both add a
    lane's cells (eight rows of eight at most) in FP32 and everything above in double-floats,
    so each is within 64 u of the sum of the magnitudes; the magnitudes of the momenta are at
    most rho / 3 here."""
    from paper_2603_13618_gb300 import inputs

    kw = dict(precision="fp16dev", tau=0.6, record=("kl",))
    batch = kss.Batch([dict(nx=nx, ny=ny)], **kw)
    batch.set_tuning(ctas_per_sm=1, multi_step=0)
    with kss.Lattice(nx, ny, **kw) as lat:
        for x in (lat, batch[0]):
            x.set_fields(*inputs.smooth_jump(nx, ny, seed=7, kmax=2))
            x.step(3) if x is lat else batch.step(3)
        a, b = lat.read_stats()[0], batch[0].read_stats()[0]
        assert np.all(np.abs(a - b) <= 2 * 64 * 2.0 ** -24 * abs(b[0])), (a, b)
    batch.close()


# ---- multi-step launches of a lone lattice against single steps ----
@pytest.mark.parametrize("precision,nx,ny", [("fp32", 1537, 1203), ("fp32", 2051, 1037),
                                             ("fp64", 515, 719), ("fp64", 515, 445)])
@pytest.mark.parametrize("switch", ["neq", "qe", None])
def test_multi_step_launch_of_ragged_lattices(kss, sms, precision, nx, ny, switch):
    """Ragged widths, partial last blocks, the seam of an odd width.  switch: the sensor that
    switches the collision of a two-relaxation lattice (None: BGK); a block then reads the
    region that its own block wrote at the step before, possibly in another CTA."""
    from paper_2603_13618_gb300 import inputs

    n = blocks(precision, nx, ny)
    assert not splits(precision, n, 32, sms)
    if precision == "fp32":
        assert n > 2 * sms
    else:  # (FP64 lattices of at most one block per SM take a launch per step)
        assert n > sms if ny == 719 else n <= sms
    fields = inputs.smooth_jump(nx, ny, seed=nx, kmax=6)
    kw = dict(precision=precision, tau=0.62, record=("kl",) if switch is None else ("kl", "qe"))
    if switch:
        kw.update(tau2=1.4, switch_sensor=switch)
        with kss.Lattice(nx, ny, **kw) as lat:  # a threshold that about half the cells pass
            lat.set_fields(*fields)
            lat.step(2)
            kw["switch_threshold"] = float(np.median(lat.read_sensor(switch)))
    a, b = kss.Lattice(nx, ny, **kw), kss.Lattice(nx, ny, **kw)
    for x in (a, b):
        x.set_fields(*fields)
        if switch:
            x.set_aar_region(inputs.random_region(nx, ny, seed=3))
    for steps in (5, 2):
        a.step(steps)
        for _ in range(steps):
            b.step(1)
        assert_equal(outputs(a), outputs(b))
        if switch:
            region = a.get_aar_region()
            assert 0 < region.sum() < nx * ny
            np.testing.assert_array_equal(region, b.get_aar_region())
            np.testing.assert_array_equal(a.read_sensor("qe"), b.read_sensor("qe"))
    a.close()
    b.close()


@pytest.mark.parametrize("nx,ny", [(33, 4987), (1, 4900), (20011, 17), (38000, 1), (765, 832)])
@pytest.mark.parametrize("tau2", [0.0, 1.4])
def test_long_runs_of_strips(kss, sms, nx, ny, tau2):
    """FP32 lattices of one row of blocks, or tall ones of slightly more blocks than SMs: runs of
    8 steps and more are one multi-step launch, shorter ones a launch per step."""
    from paper_2603_13618_gb300 import inputs

    n = blocks("fp32", nx, ny)
    assert sms < n <= 2 * sms and not splits("fp32", n, 32, sms)
    assert -(-ny // 32) == 1 or (8 * n <= 9 * sms and -(-ny // 32) >= 4 * -(-nx // 128))
    fields = inputs.smooth_jump(nx, ny, seed=9, kmax=1)
    kw = dict(precision="fp32", tau=0.62, record=("kl",), tau2=tau2)
    a, b = kss.Lattice(nx, ny, **kw), kss.Lattice(nx, ny, **kw)
    for x in (a, b):
        x.set_fields(*fields)
    for steps in (9, 7, 8):
        a.step(steps)
        for _ in range(steps):
            b.step(1)
        assert_equal(outputs(a), outputs(b))
        if tau2:
            np.testing.assert_array_equal(a.get_aar_region(), b.get_aar_region())
    a.close()
    b.close()


# ---- multi-step launches of a batch against one launch per step ----
MEMBERS = [dict(nx=37, ny=21, tau=0.7), dict(nx=130, ny=67, tau=1.0), dict(nx=1, ny=5, tau=0.8),
           dict(nx=200, ny=9, tau=0.6), dict(nx=1021, ny=1037, tau=0.9), dict(nx=5, ny=1, tau=1.3),
           dict(nx=64, ny=64, tau=0.55)]


def _member_fields(k):
    from paper_2603_13618_gb300 import inputs

    return inputs.smooth_jump(MEMBERS[k]["nx"], MEMBERS[k]["ny"], seed=30 + k, kmax=3)


@pytest.mark.parametrize("precision", ["fp32", "fp64", "fp16dev"])
@pytest.mark.parametrize("rows", [16, 32, 64])
def test_multi_step_batch_of_ragged_members(kss, sms, precision, rows):
    n = sum(blocks(precision, m["nx"], m["ny"], rows) for m in MEMBERS)
    assert not splits(precision, n, rows, sms)
    tunings = [dict(multi_step=1), dict(multi_step=0), dict(multi_step=0, ctas_per_sm=1)]
    batches = []
    for t in tunings:
        b = kss.Batch(MEMBERS, precision=precision, record=("kl",))
        b.set_tuning(rows=rows, **t)
        for k in range(len(MEMBERS)):
            b[k].set_fields(*_member_fields(k))
        batches.append(b)
    for steps in (5, 1, 4):
        for b in batches:
            b.step(steps)
        for k in range(len(MEMBERS)):
            want = outputs(batches[1][k])
            assert_equal(outputs(batches[0][k]), want)
            assert_equal(outputs(batches[2][k]), want)
    for b in batches:
        b.close()


def test_autotune_times_the_multi_step_launch(kss, sms, tmp_path):
    """The multi-step candidate is really launched (no height splits), and the states are as
    they were."""
    for rows in (16, 32, 64):
        assert not splits("fp32", sum(blocks("fp32", m["nx"], m["ny"], rows) for m in MEMBERS),
                          rows, sms)
    a = kss.Batch(MEMBERS, precision="fp32", record=("kl",))
    b = kss.Batch(MEMBERS, precision="fp32", record=("kl",))
    for k in range(len(MEMBERS)):
        for x in (a, b):
            x[k].set_fields(*_member_fields(k))
    t = a.autotune(str(tmp_path / "tune.txt"), steps=4)
    assert t["multi_step"] in (0, 1) and t["ms_per_step"] > 0
    b.set_tuning(rows=t["rows"], ctas_per_sm=1, multi_step=0)
    for k in range(len(MEMBERS)):
        np.testing.assert_array_equal(a[k].get_populations(), b[k].get_populations())
    a.step(6)
    b.step(6)
    for k in range(len(MEMBERS)):
        assert_equal(outputs(a[k]), outputs(b[k]))
    a.close()
    b.close()


@pytest.mark.parametrize("precision,nx,ny", [("fp32", 20011, 17), ("fp32", 33, 4987),
                                             ("fp64", 515, 445), ("fp64", 600, 320)])
@pytest.mark.parametrize("long_before", [False, True])
def test_long_runs_under_capture(kss, precision, nx, ny, long_before):
    """A run recorded into the caller's graph equals the call, whether or not the lattice has
    taken a run of that length before (whose workspace could not be made under capture)."""
    import torch
    from paper_2603_13618_gb300 import inputs

    fields = inputs.smooth_jump(nx, ny, seed=9, kmax=1)
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        a = kss.Lattice(nx, ny, precision=precision, tau=0.6, record=("kl",))
        b = kss.Lattice(nx, ny, precision=precision, tau=0.6, record=("kl",))
        for x in (a, b):
            x.set_fields(*fields)
            x.step(10 if long_before else 3)
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            a.step(10)
        graph.replay()
        b.step(10)
        assert_equal(outputs(a), outputs(b))
        a.close()
        b.close()
