"""GPU: output steps whose blocks are shared out to the CTAs of a cluster (small lattices)
against the same lattice in a batch, whose blocks are one CTA's each: populations, sensors,
flags, tile counts, tag counts and sums bit for bit, for every storage type and tile, at
heights around a rank's rows and a block's, and with cells that take the exact recomputation
(the density step)."""
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


def _outputs(lat, sums=True):
    flags, tiles, counts = lat.read_flags()
    out = [flags, tiles, counts, lat.get_populations(), lat.read_sensor("kl"),
           lat.read_sensor("kn")]
    return out + ([lat.read_stats()[0]] if sums else [])


@pytest.mark.parametrize("precision", ["fp32", "fp64", "fp16dev"])
@pytest.mark.parametrize("tile", [8, 16, 32, 64])
@pytest.mark.parametrize("nx,ny", [(1, 1), (33, 2), (128, 8), (130, 31), (257, 33), (300, 65)])
def test_split_steps_equal_one_cta_per_block(kss, precision, tile, nx, ny):
    from paper_2603_13618_gb300 import inputs

    fields = inputs.smooth_jump(nx, ny, seed=5, kmax=2)
    kw = dict(precision=precision, tau=0.56, tile=tile, record=("kl",))
    batch = kss.Batch([dict(nx=nx, ny=ny)], **kw)
    with kss.Lattice(nx, ny, **kw) as lat:
        for x in (lat, batch[0]):
            x.set_fields(*fields)
        for steps in (1, 4):
            lat.step(steps)
            batch.step(steps)
            # (a lone FP16 lattice adds its sums over 256-column blocks)
            for a, b in zip(_outputs(lat, precision != "fp16dev"),
                            _outputs(batch[0], precision != "fp16dev")):
                np.testing.assert_array_equal(a, b)
    batch.close()


@pytest.mark.parametrize("precision,nx,ny,record", [
    ("fp32", 501, 801, ("kl",)), ("fp32", 512, 800, ("kl", "s")), ("fp16dev", 1021, 805, ("kl",))])
def test_split_steps_of_two_rows_per_warp(kss, precision, nx, ny, record):
    """Lattices of about 100 blocks: a rank's warps take two rows each."""
    from paper_2603_13618_gb300 import inputs

    fields = inputs.smooth_jump(nx, ny, seed=6, kmax=3)
    kw = dict(precision=precision, tau=0.6, record=record)
    batch = kss.Batch([dict(nx=nx, ny=ny)], **kw)
    with kss.Lattice(nx, ny, **kw) as lat:
        for x in (lat, batch[0]):
            x.set_fields(*fields)
            x.step(3) if x is lat else batch.step(3)
        for a, b in zip(_outputs(lat, precision != "fp16dev"),
                        _outputs(batch[0], precision != "fp16dev")):
            np.testing.assert_array_equal(a, b)
    batch.close()


@pytest.mark.parametrize("precision", ["fp32", "fp64", "fp16dev"])
@pytest.mark.parametrize("record,switch,at", [(("kl",), "neq", 1e-3), (("hr", "s"), "qe", 1e-5)])
def test_split_two_relaxation_steps(kss, precision, record, switch, at):
    """The two-relaxation step, fused and all-sensor, its region included.  (A batch takes
    the all-sensor step for a qe switch, a lone lattice the fused one: so neq there.)"""
    from paper_2603_13618_gb300 import inputs

    nx, ny = 270, 70
    fields = inputs.smooth_jump(nx, ny, seed=8, kmax=3)
    kw = dict(precision=precision, tau=0.7, tau2=1.4, record=record, switch_sensor=switch,
              switch_threshold=at)
    batch = kss.Batch([dict(nx=nx, ny=ny)], **kw)
    with kss.Lattice(nx, ny, **kw) as lat:
        for x in (lat, batch[0]):
            x.set_fields(*fields)
        lat.step(5)
        batch.step(5)
        for a, b in zip(_outputs(lat) + [lat.get_aar_region()],
                        _outputs(batch[0]) + [batch[0].get_aar_region()]):
            np.testing.assert_array_equal(a, b)
    batch.close()


@pytest.mark.parametrize("precision", ["fp32", "fp64", "fp16dev"])
@pytest.mark.parametrize("rows", [16, 32, 64])
@pytest.mark.parametrize("shapes", [[(1, 1)], [(64, 64), (33, 17), (200, 90)],
                                    [(128, 65)] * 7, [(300, 64), (129, 1), (128, 33), (5, 200)]])
def test_split_batches_equal_one_cta_per_block(kss, precision, rows, shapes):
    """Batches with few blocks, against the same batch with persistent CTAs (one per block);
    the second set's sums are those of the last step of each run."""
    from paper_2603_13618_gb300 import inputs

    kw = dict(precision=precision, tau=0.56, record=("kl",), output_every=1)
    a = kss.Batch([dict(nx=nx, ny=ny) for nx, ny in shapes], **kw)
    b = kss.Batch([dict(nx=nx, ny=ny) for nx, ny in shapes], **kw)
    a.set_tuning(rows=rows)
    b.set_tuning(rows=rows, ctas_per_sm=1, multi_step=0)
    for k, (nx, ny) in enumerate(shapes):
        fields = inputs.smooth_jump(nx, ny, seed=20 + k, kmax=2)
        a[k].set_fields(*fields)
        b[k].set_fields(*fields)
    for steps in (1, 5, 2):
        a.step(steps)
        b.step(steps)
        for x, y in zip(a.members, b.members):
            for u, v in zip(_outputs(x), _outputs(y)):
                np.testing.assert_array_equal(u, v)
    a.close()
    b.close()


@pytest.mark.parametrize("nx,ny", [(64, 64), (300, 200), (900, 1000)])
def test_runs_under_capture(kss, nx, ny):
    """A run of output steps recorded into the caller's graph: one replay equals the call."""
    import torch
    from paper_2603_13618_gb300 import inputs

    fields = inputs.smooth_jump(nx, ny, seed=9, kmax=2)
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        a = kss.Lattice(nx, ny, precision="fp32", tau=0.6, record=("kl",))
        b = kss.Lattice(nx, ny, precision="fp32", tau=0.6, record=("kl",))
        for x in (a, b):
            x.set_fields(*fields)
            for _ in range(3):
                x.step(4)
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            a.step(4)
        graph.replay()
        b.step(4)
        for u, v in zip(_outputs(a), _outputs(b)):
            np.testing.assert_array_equal(u, v)
        a.close()
        b.close()
