"""The estimator on grids and widths that take every form of its layers: levels
that tile into rows, part rows or not at all, channel counts that are and are
not multiples of 32, batches of one and of several.  Forward within 2e-3 and
gradients within 2e-2 (relative norm per layer) of the FP64 oracle that rounds
to BF16 where the GPU stores BF16, as in the parity tests; a second backward
pass gives the same gradients bit for bit."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import cnn as ocnn  # noqa: E402


@pytest.fixture(scope="module")
def gd():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1204_6367_gb300 import build, gdrr
    build.build()
    gdrr.lib()
    return gdrr


def _rel(a, b):
    return np.linalg.norm(a - b) / max(np.linalg.norm(b), 1e-30)


@pytest.mark.parametrize("c, H, W, B", [(8, 8, 8, 1), (24, 16, 24, 2), (32, 64, 64, 1), (32, 40, 128, 2), (48, 32, 32, 1),
                                        (64, 32, 64, 1), (32, 16, 256, 1), (16, 32, 128, 3), (32, 8, 128, 1), (32, 24, 48, 2),
                                        (32, 24, 40, 3), (32, 8, 136, 2)])
def test_forward_and_gradients(gd, c, H, W, B):
    rng = np.random.default_rng(c * H + W)
    flat = ocnn.init_params(c, c + H).astype(np.float32)
    x = rng.normal(size=(B, 2, H, W)).astype(np.float32)
    t = rng.normal(size=(B, 1, H, W)).astype(np.float32)
    net = gd.Cnn(B, H, W, c)
    net.set_params(flat)
    xb, tb = torch.from_numpy(x).cuda(), torch.from_numpy(t).cuda()
    out = net.forward(xb).cpu().numpy()
    loss = net.backward(tb)
    grads = net.get_grads()
    net.forward(xb)
    net.backward(tb)
    np.testing.assert_array_equal(net.get_grads(), grads)
    net.close()
    ref, cache = ocnn.forward(x, flat.astype(np.float64), c)
    rloss, rgrads = ocnn.backward(cache, t)
    assert _rel(out, ref) < 2e-3
    assert abs(loss - rloss) < 1e-3 * abs(rloss)
    off = 0
    for ci, co, k, _ in ocnn.specs(c):
        for n in (co * ci * k * k, co):
            assert _rel(grads[off:off + n], rgrads[off:off + n]) < 2e-2, (ci, co, n)
            off += n
