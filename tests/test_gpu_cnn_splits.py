"""Weight gradients of 256 output channels on grids that do not tile (10 x 6 pixels,
69 images: 4140 pixels): the column form's product, in pairs of CTAs with its pixels
split, is summed in order.  Gradients within 2e-2 (relative norm per
layer) of the FP64 oracle that rounds to BF16 where the GPU stores BF16, and the
same bits in a second pass."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import cnn as ocnn  # noqa: E402


def test_split_column_product_in_pairs():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1204_6367_gb300 import build, gdrr
    build.build()
    c, B, H, W = 64, 69, 40, 24
    rng = np.random.default_rng(7)
    flat = ocnn.init_params(c, 3).astype(np.float32)
    x = rng.normal(size=(B, 2, H, W)).astype(np.float32)
    t = rng.normal(size=(B, 1, H, W)).astype(np.float32)
    net = gdrr.Cnn(B, H, W, c)
    net.set_params(flat)
    xb, tb = torch.from_numpy(x).cuda(), torch.from_numpy(t).cuda()
    net.forward(xb)
    net.backward(tb)
    grads = net.get_grads()
    net.forward(xb)
    net.backward(tb)
    np.testing.assert_array_equal(net.get_grads(), grads)
    net.close()
    _, cache = ocnn.forward(x, flat.astype(np.float64), c)
    _, ref = ocnn.backward(cache, t)
    off = 0
    for ci, co, k, _ in ocnn.specs(c):
        for n in (co * ci * k * k, co):
            assert np.linalg.norm(grads[off:off + n] - ref[off:off + n]) < 2e-2 * np.linalg.norm(ref[off:off + n]), (ci, co, n)
            off += n
