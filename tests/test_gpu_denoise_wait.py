"""A denoiser tile whose neighbour is not there gives up: after the limit it is
given and not much later, with the timeout's code and its output unwritten, and
the next denoiser call on the same stream gives the per-iteration form's bits."""
import time

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1204_6367_gb300 import inputs  # noqa: E402


@pytest.mark.parametrize("limit_ms", [1, 20, 200])
def test_a_tile_without_its_neighbour_gives_up(limit_ms):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1204_6367_gb300 import build, gdrr
    build.build()
    gdrr.gdrr_probe_bounded_wait(1)                      # first launch: code is loaded
    t0 = time.perf_counter()
    assert gdrr.gdrr_probe_bounded_wait(limit_ms * 1_000_000) == -7
    took = time.perf_counter() - t0
    assert limit_ms * 1e-3 <= took < limit_ms * 1e-3 + 0.2
    s = torch.linspace(10.0, 40.0, 96 * 128, dtype=torch.float64, device="cuda").reshape(96, 128)
    with gdrr.Context(inputs.small_problem()) as ctx:
        got = gdrr.gdrr_denoise_scatter(ctx, s, 1.0, 0.05, iters=30)
        gdrr.gdrr_sync(ctx)
    assert torch.equal(got, gdrr.gdrr_denoise_scatter_static(s, 1.0, 0.05, iters=30))
