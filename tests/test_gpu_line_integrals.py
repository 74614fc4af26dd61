"""The line integrals against the logarithm in 64 bits where its value is most
exposed: signal and air close to each other on either side of a power of two,
and ratios all over [1/2, 2].  For such a ratio s - a is exact in FP64 and
log1p((s - a) / a) is good to 2^-51 relative (a division and a logarithm of at
most 2 ulp), 2^-27 of an FP32 ulp: a value that is the FP32 rounding of the
logarithm lies within 0.5 + 2^-26 ulp of it, and the tests allow 0.5 + 2^-20."""
import numpy as np
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


def _ulps(gd, sig, air):
    """Distance from the logarithm in FP32 ulps of the result (sig [views, n], air [n])."""
    got = gd.gdrr_line_integrals_views(torch.from_numpy(sig).cuda(), torch.from_numpy(air).cuda(), 1e-6).cpu().numpy()
    exact = -np.log1p((sig - air) / air)
    ulp = np.spacing(np.maximum(np.abs(got), np.finfo(np.float32).tiny)).astype(np.float64)
    return np.abs(got.astype(np.float64) - exact) / ulp


@pytest.mark.parametrize("gap", [1e-9, 1e-7, 1e-6, 1e-5, 1e-4, 1e-3])
@pytest.mark.parametrize("power", [2.0 ** -30, 1.0, 2.0, 4.0])
def test_signal_and_air_on_either_side_of_a_power_of_two(gd, gap, power):
    rng = np.random.default_rng(int(-np.log10(gap)))
    below = power * (1.0 - gap * rng.uniform(0.01, 1.0, 20_000))
    above = power * (1.0 + gap * rng.uniform(0.01, 1.0, (9, 20_000)))
    assert _ulps(gd, above, below).max() <= 0.5 + 2.0 ** -20
    swapped = power * (1.0 - gap * rng.uniform(0.01, 1.0, (9, 20_000)))
    assert _ulps(gd, swapped, above[0]).max() <= 0.5 + 2.0 ** -20


@pytest.mark.parametrize("lo, hi", [(0.5, 0.7072), (0.7071, 0.9), (0.9, 1.1), (1.1, 1.4143), (1.4142, 2.0)])
def test_ratios_of_every_size(gd, lo, hi):
    rng = np.random.default_rng(int(1000 * lo))
    air = np.exp(rng.uniform(-25.0, 3.0, 200_003))
    sig = air[None] * rng.uniform(lo, hi, (10, 200_003))
    sig = np.clip(sig, 0.5 * air, 2.0 * air)
    assert _ulps(gd, sig, air).max() <= 0.5 + 2.0 ** -20
