"""The GEMM's paired form at the edges of its 256 x 256 tiles, with and without K
splits, against FP64, and the form that it replaces (a row of C that is not a
multiple of 16 bytes) bit for bit.  A product step of 16 truncates its sum at
24 bits, so K / 16 steps stay within K / 16 * 2^-22 of the exact result
(relative norm)."""
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


def _operands(m, n, k):
    g = torch.Generator(device="cuda").manual_seed(m * n + k)
    return (torch.randn((m, k), device="cuda", generator=g).bfloat16(),
            torch.randn((n, k), device="cuda", generator=g).bfloat16())


@pytest.mark.parametrize("m, n, k", [(129, 256, 64), (256, 260, 192), (257, 512, 1024), (300, 1000, 448), (640, 776, 64),
                                     (2047, 2304, 320)])
def test_tile_edges(gd, m, n, k):
    a, b = _operands(m, n, k)
    ref = a.double() @ b.double().T
    c = gd.gdrr_gemm_bf16(a, b)
    assert (c.double() - ref).norm() <= k / 16 * 2.0 ** -22 * ref.norm()


@pytest.mark.parametrize("m, n, k", [(129, 258, 64), (300, 513, 640), (515, 1022, 1024)])
def test_same_bits_as_single_cta_form(gd, m, n, k):
    # a row of n floats is no multiple of 16 bytes: the single-CTA form
    a, b = _operands(m, (n + 3) // 4 * 4, k)
    assert n % 4
    torch.testing.assert_close(gd.gdrr_gemm_bf16(a, b[:n].contiguous()), gd.gdrr_gemm_bf16(a, b)[:, :n], rtol=0, atol=0)
