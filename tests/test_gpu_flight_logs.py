"""The free flights' logarithm takes its quotient from an approximate reciprocal
and a residual correction.  For every 24-bit uniform it equals the oracle's, which
divides: all 2^24 values, bit for bit."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle  # noqa: E402


@pytest.mark.gpu
def test_every_uniform():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1204_6367_gb300 import build, gdrr
    build.build()
    got = gdrr.gdrr_flight_logs(1, 1 << 24).cpu().numpy()
    k = np.arange(1, (1 << 24) + 1)
    ref = oracle.logf((k * 2.0 ** -24).astype(np.float32))
    np.testing.assert_array_equal(got.view(np.uint32), ref.view(np.uint32))
    np.testing.assert_array_equal(gdrr.gdrr_flight_logs(77, 300).cpu().numpy(), ref[76:376])


def test_arguments_are_checked():
    from paper_1204_6367_gb300 import build, gdrr
    build.build()
    for k0, n in ((0, 1), (1, -1), ((1 << 24) + 1, 1), (1, (1 << 24) + 1), (1, 5)):
        assert gdrr.lib().gdrr_flight_logs(k0, n, None, None) == -1
