"""The tri-linear ray tracer at ragged detector sizes, odd phantoms and other
material counts, against the oracle's FP64 trace (rtol 2e-4: FP32 path sums of
up to a thousand midpoints and positions good to 1e-4 mm, as in the parity
tests)."""
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


def _check(gd, prob, phi):
    with gd.Context(prob) as ctx:
        P = gd.gdrr_raytrace_primary(ctx, phi).cpu().numpy()
    ref = oracle.rt_primary(prob, phi=phi)
    np.testing.assert_allclose(P, ref, rtol=2e-4, atol=1e-12 * ref.max())


@pytest.mark.parametrize("nu, nv", [(1, 1), (17, 9), (33, 5), (16, 8), (3, 40)])
def test_ragged_detectors(gd, nu, nv):
    _check(gd, inputs.torso_problem(vox=8.0, nu=nu, nv=nv, det_px=300.0 / max(nu, nv)), 0.9)


@pytest.mark.parametrize("labels", [2, 3, 8])
def test_mixed_labels_of_one_material(gd, labels):
    # voxels of one substance under several material indices: the same field,
    # summed per index, so only the FP32 summation order differs (at most 8 x 40
    # terms of a path integral below 2: 320 x 2^-24 x 2 < 5e-5 of the signal)
    rng = np.random.default_rng(labels)
    p = inputs.uniform_slab_problem(nx=13, ny=1, nz=7, nu=12, nv=10, det_px=2.0, pencil=False,
                                    materials=[inputs.WATER] * labels)
    p.density[:] = rng.uniform(0.0, 2.0, p.density.shape)
    out = []
    for mixed in (False, True):
        p.material[:] = rng.integers(0, labels, p.material.shape) if mixed else 0
        with gd.Context(p) as ctx:
            out.append([gd.gdrr_raytrace_primary(ctx, phi).cpu().numpy() for phi in (0.0, 0.4, 1.6)])
    np.testing.assert_allclose(out[1], out[0], rtol=5e-5)
