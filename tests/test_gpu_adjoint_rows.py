"""GPU: the reverse step's rows per warp.  A lattice tiled from copies of a smaller periodic
one has the smaller one's gradient in every copy, cell by cell the same arithmetic, so the
two agree bit for bit although the large one's warps take two or four rows each; J and dJ/dtau
are the copies' sum (their partial sums are formed in another order: 1e-6 of them in FP32).
Also the order of calls: forward passes without a backward one, and a changed tau."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,copies", [(220, 7), (222, 10)])
def test_tiled_lattice_has_the_tiled_gradient(n, copies):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2603_13618_gb300 import inputs, kss

    small = inputs.random_smooth(n, n, seed=12, kmax=3)
    large = [np.tile(a, (copies, copies)) for a in small]
    with kss.Adjoint(n, n, 7, checkpoint_every=3) as a, \
            kss.Adjoint(n * copies, n * copies, 7, checkpoint_every=3) as b:
        for tau in (0.6, 0.9):
            ja = a.forward(*small, tau)
            if tau == 0.9:  # forward passes alone, then one with its backward pass
                a.forward(*small, 0.7)
                a.forward(*small, 0.7)
                assert a.forward(*small, tau) == ja
            ga, ta = a.backward()
            jb = b.forward(*large, tau)
            gb, tb = b.backward()
            np.testing.assert_array_equal(gb, np.tile(ga, (copies, copies)))
            assert jb == pytest.approx(ja * copies ** 2, rel=1e-6)
            assert tb == pytest.approx(ta * copies ** 2, rel=1e-5)
