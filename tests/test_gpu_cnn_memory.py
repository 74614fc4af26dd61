"""What a network holds: its activations (BF16), the gradients a pass reads (FP32:
of the concatenated decoder inputs and the pooled encoder inputs), one dZ (BF16),
one row of 32 tap values per pixel (BF16), the weight gradients' partial sums
(FP32, one per 4096 pixels and layer), and the weights with their gradients,
moments and copies.  Where no layer needs a column matrix none is held."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gd():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1204_6367_gb300 import build, gdrr
    build.build()
    gdrr.lib()
    return gdrr


def _held(gd, B, H, W, c):
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    net = gd.Cnn(B, H, W, c)
    held = before - torch.cuda.mem_get_info()[0]
    net.close()
    return held


@pytest.mark.parametrize("B, H, W, c", [(64, 96, 128, 32), (24, 128, 128, 64), (32, 64, 256, 32)])
def test_no_column_buffers_where_no_layer_uses_them(gd, B, H, W, c):
    gd.Cnn(1, H, W, c).close()                                 # the context's own allocations
    s1 = B * H * W
    s2, s3, s4 = s1 // 4, s1 // 16, s1 // 64
    cats = 3 * c * s1 + 6 * c * s2 + 12 * c * s3               # concatenated decoder inputs
    pooled = c * s2 + 2 * c * s3 + 4 * c * s4                  # pooled encoder inputs
    need = 2 * (2 * s1 + cats + pooled + c * s1) + 4 * s1      # activations and the output
    need += 4 * (cats + pooled)                                # their gradients
    need += 2 * c * s1 + 2 * 32 * s1                           # dZ, tap rows
    for level, ci, co in ((0, 2, c), (1, c, 2 * c), (2, 2 * c, 4 * c), (3, 4 * c, 8 * c), (2, 12 * c, 4 * c),
                          (1, 6 * c, 2 * c), (0, 3 * c, c)):
        need += 4 * ((s1 >> 2 * level) // 4096 + 1) * co * max(32, 9 * ci) + (4 * 4 + 2 * 2) * 9 * ci * co
    assert _held(gd, B, H, W, c) <= 1.1 * need + (100 << 20)
