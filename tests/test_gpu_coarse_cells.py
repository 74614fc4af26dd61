"""The global majorant in coarse macro cells, which decides its collisions in the
flight: tallies and counters equal the CPU oracle's exactly, and as many collisions
are virtual by their cell's bound as in a run with event records, which tests the
bound first."""
import os

import numpy as np
import pytest
import torch

import oracle
from paper_1204_6367_gb300 import inputs

pytestmark = pytest.mark.gpu
NTH = os.cpu_count() or 1


@pytest.fixture(scope="module")
def gd():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1204_6367_gb300 import build, gdrr
    build.build()
    gdrr.lib()
    return gdrr


def _problem(vox, n_mat):
    if n_mat == 4:
        p = inputs.torso_problem(vox=vox, nu=40, nv=30, det_px=9.9)
        p.material = np.ascontiguousarray(p.material[:, 3:, 5:])      # ragged
        p.density = np.ascontiguousarray(p.density[:, 3:, 5:])
        return p
    mats = [inputs.AIR, inputs.BONE, inputs.WATER, inputs.LUNG, inputs.ALUMINIUM, inputs.WATER, inputs.BONE, inputs.LUNG]
    p = inputs.uniform_slab_problem(nx=21, ny=18, nz=17, vox=vox, nu=16, nv=16, det_px=9.0, pencil=False,
                                    materials=mats[:n_mat])
    p.material[:] = (np.arange(21) // 5 % n_mat).astype(np.uint8)[None, None, :]
    p.density[:] = np.random.default_rng(3).uniform(0.0, 1.8, p.density.shape)
    p.form_factor = None
    return p


@pytest.mark.parametrize("vox, shift, n_mat", [(8.0, 4, 4), (8.0, 5, 4), (16.0, 3, 4), (16.0, 6, 4), (16.0, 3, 2), (32.0, 2, 8),
                                               (8.0, 3, 4)])               # 64 mm: by way of the gather service
@pytest.mark.parametrize("opts", [{}, {"max_steps": 7}, {"scatter_filter": 3}, {"rayleigh_form_factor": 1}])
def test_same_events_and_counts(gd, vox, shift, n_mat, opts):
    prob, n = _problem(vox, n_mat), 20_011
    if "rayleigh_form_factor" in opts and prob.form_factor is None:
        pytest.skip("no form factors")
    names = {"rayleigh_form_factor": "rayleigh_ff"}
    ref = oracle.mc_run(prob, n, seed=4, phi=0.7, angle_index=3, threads=NTH,
                        **{names.get(k, k): (bool(v) if k in names else v) for k, v in opts.items()})
    skips = []
    with gd.Context(prob) as ctx:
        gd.gdrr_set_options(ctx, cell_shift=shift, **opts)
        for records in (False, True):
            st = torch.zeros(gd.GDRR_NSTATS, dtype=torch.int64, device="cuda")
            rec = torch.zeros(n * gd.RECORD_DTYPE.itemsize, dtype=torch.uint8, device="cuda") if records else None
            p, s = gd.gdrr_mc_project(ctx, n, 4, 0.7, 3, stats=st, records=rec)
            gd.gdrr_sync(ctx)
            assert gd.stats_dict(st) == ref[2]
            np.testing.assert_array_equal(p.cpu().numpy(), ref[0])
            np.testing.assert_array_equal(s.cpu().numpy(), ref[1])
            skips.append(int(gd.cell_skips(st)))
    assert skips[0] == skips[1] > 0
