"""The ray trace sums a ray's densities into one running sum while its samples
are of one material and into one per material where they mix.  Both add the same
terms in the same order: voxels of zero density add nothing whatever their
label, so labelling them as another material (which sends most samples the mixed
way) leaves every pixel as it is, to the bit."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1204_6367_gb300 import inputs  # noqa: E402

MATERIALS = [inputs.AIR, inputs.WATER, inputs.BONE, inputs.LUNG, inputs.ALUMINIUM, inputs.WATER, inputs.BONE, inputs.LUNG]


@pytest.mark.parametrize("n_mat", [2, 4, 8])
@pytest.mark.parametrize("empty", [0.03, 0.3, 0.9])
def test_labels_of_empty_voxels_change_nothing(n_mat, empty):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1204_6367_gb300 import build, gdrr
    build.build()
    rng = np.random.default_rng(n_mat)
    out = []
    shape = (23, 31, 29)
    density = rng.uniform(0.2, 2.0, shape) * (rng.uniform(size=shape) >= empty)
    labels = rng.integers(0, n_mat, shape)
    for relabel in (False, True):
        p = inputs.uniform_slab_problem(nx=29, ny=31, nz=23, nu=70, nv=50, det_px=1.7, pencil=False,
                                        materials=MATERIALS[:n_mat])
        p.density[:] = density
        p.material[:] = np.where((density == 0.0) & relabel, labels, 1)
        p.form_factor = None
        with gdrr.Context(p) as ctx:
            out.append(np.stack([gdrr.gdrr_raytrace_primary(ctx, a).cpu().numpy() for a in (0.0, 0.4, 1.57, 3.9)]))
    assert np.ptp(out[0]) > 0
    np.testing.assert_array_equal(out[0], out[1])
