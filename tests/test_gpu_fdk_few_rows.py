"""The row filter on few rows, where several blocks share them, and in place,
where none may: against FP64 (at most nu / 2 products of magnitude up to max|q| /
(2 tau), each rounded within 2^-24: 1e-5 max|g| / tau bounds the sum), and the
same bits either way."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import fdk as ofdk  # noqa: E402


@pytest.fixture(scope="module")
def gd():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1204_6367_gb300 import build, gdrr
    build.build()
    gdrr.lib()
    return gdrr


@pytest.mark.parametrize("nu, nv, n", [(1, 1, 1), (8, 8, 1), (64, 48, 16), (512, 1, 1), (777, 3, 2), (1030, 10, 1), (2048, 2, 2),
                                       (4096, 1, 1), (4095, 8, 16)])
def test_few_rows_and_in_place(gd, nu, nv, n):
    rng = np.random.default_rng(nu + n)
    sad, sdd, du, dv = 1000.0, 1500.0, 0.9, 1.1
    g = rng.uniform(0.0, 3.0, (n, nv, nu)).astype(np.float32)
    geo = gd.fdk_geometry(sad, sdd, nu, nv, du, dv, (4, 4, 4), (1.0, 1.0, 1.0))
    got = gd.gdrr_fdk_filter(geo, torch.from_numpy(g).cuda())
    ref = ofdk.fdk_filter(g.astype(np.float64), sad, sdd, du, dv)
    np.testing.assert_allclose(got.cpu().numpy(), ref, rtol=0, atol=1e-5 * float(np.abs(g).max()) / (du * sad / sdd))
    x = torch.from_numpy(g).cuda()
    gd.gdrr_fdk_filter(geo, x, out=x)
    assert torch.equal(x, got)
