"""Volumes of more slices than one launch has blocks for (65535 in z, four
slices each): reconstructed as the oracle does, in FP32 (positions good to 1e-5
pixel and n_views rounded sums, 1e-4 of the largest magnitude)."""
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


@pytest.mark.parametrize("nz", [262_140, 262_143, 524_287, 700_001])
@pytest.mark.parametrize("accumulate", [False, True])
def test_more_slices_than_blocks_in_z(gd, nz, accumulate):
    rng = np.random.default_rng(nz)
    sad, sdd, nu, nv, du, dv = 900.0, 1400.0, 8, 32, 2.5, 2.5
    shape, vox = (nz, 1, 2), (1.0, 1.0, 80.0 / nz)         # the column spans the detector's rows and more
    angles = np.sort(rng.uniform(0.0, 6.28, 5))
    q = rng.normal(0.0, 1.0, (5, nv, nu)).astype(np.float32)
    geo = gd.fdk_geometry(sad, sdd, nu, nv, du, dv, shape, vox)
    vol = torch.full(shape, 0.25, device="cuda") if accumulate else None
    got = gd.gdrr_fdk_backproject(geo, torch.from_numpy(q).cuda(), angles, 0.037, vol, accumulate).cpu().numpy()
    ref = ofdk.fdk_backproject(q.astype(np.float64), angles, 0.037, sad, sdd, du, dv, shape, vox) + 0.25 * accumulate
    np.testing.assert_allclose(got, ref, rtol=0, atol=1e-4 * float(np.abs(ref).max()))
