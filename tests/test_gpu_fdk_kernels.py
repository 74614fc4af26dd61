"""The reconstruction kernels at the edges of their tiles, against FP64.

Line integrals: what is written is the FP32 rounding of the FP64 logarithm, so
it lies within half an FP32 ulp (plus 2^-10 of one for the FP64 operations) of
the exact value.  Filter: at most nu / 2 products of magnitude up to max|q| / (2
tau), each rounded within 2^-24: 1e-5 max|g| / tau bounds the sum.
Backprojection: FP32 positions good to 1e-5 pixel and n_views rounded sums:
1e-4 of the largest magnitude."""
import math

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


def _half_ulp(got, ref):
    ulp = np.spacing(np.maximum(np.abs(got), np.finfo(np.float32).tiny).astype(np.float32)).astype(np.float64)
    assert np.all(np.abs(got.astype(np.float64) - ref) <= (0.5 + 2.0 ** -10) * ulp)


@pytest.mark.parametrize("spread", [1e-12, 1e-7, 1e-4, 0.02, 1.0, 12.0])
def test_line_integrals_round_the_logarithm(gd, spread):
    rng = np.random.default_rng(int(-10 * math.log10(spread)) + 50)
    air = np.exp(rng.uniform(-25.0, 3.0, 5003))
    sig = air[None] * np.exp(rng.uniform(-spread, spread, (19, 5003)))
    sig[:, ::97] = air[::97]                                   # exactly zero attenuation
    got = gd.gdrr_line_integrals_views(torch.from_numpy(sig).cuda(), torch.from_numpy(air).cuda(), 1e-6).cpu().numpy()
    x = np.longdouble(sig) / np.longdouble(air)
    # the quotient is rounded to FP64 first, which near 1 is all the value has
    q = np.log(np.maximum(sig, 1e-6 * air) / air)
    exact = -np.log(np.maximum(x, np.longdouble(1e-6)))
    tol = np.abs(np.asarray(exact - np.longdouble(-q), np.float64))
    ulp = np.spacing(np.maximum(np.abs(got), np.finfo(np.float32).tiny)).astype(np.float64)
    assert np.all(np.abs(got - np.asarray(exact, np.float64)) <= (0.5 + 2.0 ** -10) * ulp + tol)
    one = gd.gdrr_line_integrals(torch.from_numpy(sig[3]).cuda(), torch.from_numpy(air).cuda(), 1e-6).cpu().numpy()
    np.testing.assert_array_equal(one, got[3])


def test_line_integrals_of_special_values(gd):
    air = np.array([1.0, 1.0, 1.0, 1.0, 1.0, 5e-324, 1e-310, 0.0, 2.0, 1e300])
    sig = np.array([0.0, -1.0, np.nan, np.inf, 1e-320, 1.0, 1e-311, 1.0, -np.inf, 1e-300])
    got = gd.gdrr_line_integrals(torch.from_numpy(sig).cuda(), torch.from_numpy(air).cuda(), 1e-6).cpu().numpy()
    with np.errstate(all="ignore"):
        ref = (-np.log(np.fmax(sig, 1e-6 * air) / air)).astype(np.float32)
    np.testing.assert_array_equal(got, ref)


@pytest.mark.parametrize("nu, nv, n", [(1, 3, 2), (7, 5, 3), (16, 33, 2), (17, 4, 5), (255, 3, 3), (512, 9, 4),
                                       (1030, 5, 2), (4096, 3, 3)])
def test_filter_at_tile_edges(gd, nu, nv, n):
    rng = np.random.default_rng(nu)
    sad, sdd, du, dv = 1000.0, 1500.0, 0.9, 1.1
    g = rng.uniform(0.0, 3.0, (n, nv, nu)).astype(np.float32)
    geo = gd.fdk_geometry(sad, sdd, nu, nv, du, dv, (4, 4, 4), (1.0, 1.0, 1.0))
    got = gd.gdrr_fdk_filter(geo, torch.from_numpy(g).cuda()).cpu().numpy().astype(np.float64)
    ref = ofdk.fdk_filter(g.astype(np.float64), sad, sdd, du, dv)
    np.testing.assert_allclose(got, ref, rtol=0, atol=1e-5 * float(np.abs(g).max()) / (du * sad / sdd))


@pytest.mark.parametrize("shape, vox, nu, nv", [((9, 33, 35), (2.0, 2.0, 2.0), 64, 48),     # inside the detector
                                                ((17, 9, 31), (4.0, 3.0, 5.0), 37, 11),     # beyond its edges
                                                ((1, 1, 1), (1.0, 1.0, 1.0), 8, 8)])
def test_backprojection_inside_and_across_the_detector_edge(gd, shape, vox, nu, nv):
    rng = np.random.default_rng(nu)
    sad, sdd, du, dv = 900.0, 1400.0, 2.5, 2.5
    n = 33
    angles = np.sort(rng.uniform(0.0, 2.0 * math.pi, n))
    q = rng.normal(0.0, 1.0, (n, nv, nu)).astype(np.float32)
    geo = gd.fdk_geometry(sad, sdd, nu, nv, du, dv, shape, vox)
    got = gd.gdrr_fdk_backproject(geo, torch.from_numpy(q).cuda(), angles, d_beta=0.037).cpu().numpy()
    ref = ofdk.fdk_backproject(q.astype(np.float64), angles, 0.037, sad, sdd, du, dv, shape, vox)
    np.testing.assert_allclose(got, ref, rtol=0, atol=1e-4 * float(np.abs(ref).max()))
