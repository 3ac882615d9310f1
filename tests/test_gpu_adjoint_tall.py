"""GPU: the gradient of a lattice taller than 65535 blocks of the reverse step's usual rows
(16 per block: 1 048 560), tiled from copies of a short periodic one: every copy has the short
one's gradient bit for bit; J and dJ/dtau are the copies' sum (FP32 partials, 1e-5)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,rel", [("fp32", 1e-5), ("fp64", 1e-10)])
@pytest.mark.parametrize("copies", [65535, 65536])
def test_tall_lattice_has_the_tiled_gradient(precision, rel, copies):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2603_13618_gb300 import inputs, kss

    nx, n = 3, 16
    small = inputs.random_smooth(nx, n, seed=12, kmax=1)
    tall = [np.tile(a, (copies, 1)) for a in small]
    with kss.Adjoint(nx, n, 3, precision=precision, checkpoint_every=1) as a:
        ja = a.forward(*small, 0.7)
        ga, ta = a.backward()
    with kss.Adjoint(nx, n * copies, 3, precision=precision, checkpoint_every=1) as b:
        jb = b.forward(*tall, 0.7)
        gb, tb = b.backward()
    np.testing.assert_array_equal(gb, np.tile(ga, (copies, 1)))
    assert jb == pytest.approx(ja * copies, rel=rel)
    assert tb == pytest.approx(ta * copies, rel=rel)
