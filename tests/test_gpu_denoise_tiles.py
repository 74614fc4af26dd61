"""The one-launch denoiser over tile shapes: one pixel, single rows and columns,
ragged tiles, one to four pixels per thread.  It runs the per-iteration
kernel's FP64 operations in the same order, so it equals that form (the
allocation-free entry point) bit for bit; images beyond that entry point's
limit equal the CPU oracle to FP64 rounding (rtol 1e-11, the bound of the
oracle comparison at 400 iterations)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import oracle  # noqa: E402
from paper_1204_6367_gb300 import inputs  # noqa: E402


@pytest.fixture(scope="module")
def gd():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1204_6367_gb300 import build, gdrr
    build.build()
    gdrr.lib()
    return gdrr


@pytest.mark.parametrize("nu, nv", [(1, 1), (1, 77), (200, 1), (2, 3), (33, 5), (43, 97), (128, 96), (257, 152), (511, 128),
                                    (8, 4096)])
@pytest.mark.parametrize("iters", [0, 1, 2, 61])
def test_equals_the_iteration_by_launches(gd, nu, nv, iters):
    rng = np.random.default_rng(nu * 1000 + nv)
    s = torch.from_numpy(rng.poisson(30.0, (nv, nu)).astype(np.float64) * 2e-9).cuda()
    with gd.Context(inputs.small_problem()) as ctx:
        got = gd.gdrr_denoise_scatter(ctx, s, 2e-9, 0.05, iters=iters)
        again = gd.gdrr_denoise_scatter(ctx, s, 2e-9, 0.05, iters=iters)     # stale words of the first call
        gd.gdrr_sync(ctx)
    assert torch.equal(got, again)
    assert torch.equal(got, gd.gdrr_denoise_scatter_static(s, 2e-9, 0.05, iters=iters))


@pytest.mark.parametrize("nu, nv", [(512, 384), (900, 601)])
def test_large_images_match_the_oracle(gd, nu, nv):
    rng = np.random.default_rng(nu)
    s = rng.poisson(30.0, (nv, nu)).astype(np.float64)
    with gd.Context(inputs.small_problem()) as ctx:
        got = gd.gdrr_denoise_scatter(ctx, torch.from_numpy(s).cuda(), 1.0, 0.05, iters=40).cpu().numpy()
        gd.gdrr_sync(ctx)
    np.testing.assert_allclose(got, oracle.denoise(s, 0.05, 0.8, 40), rtol=1e-11)


def test_non_finite_counts_stay_where_they_are(gd):
    s = torch.full((9, 40), 20.0, dtype=torch.float64, device="cuda")
    s[3, 7] = float("nan")
    s[5, 30] = float("inf")
    with gd.Context(inputs.small_problem()) as ctx:
        got = gd.gdrr_denoise_scatter(ctx, s, 1.0, 0.05, iters=3).cpu().numpy()
        gd.gdrr_sync(ctx)
    np.testing.assert_array_equal(got, gd.gdrr_denoise_scatter_static(s, 1.0, 0.05, iters=3).cpu().numpy())
