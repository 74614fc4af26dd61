"""Runs with event records over the launch shapes that shape them (threads per
block, waiting lanes per service, histories per claim, resident blocks), and
with the coefficient tables of 8 materials at 512 threads (48 KB a block, beyond
the default shared-memory limit): records, tallies and counters equal the CPU
oracle's exactly."""
import os

import numpy as np
import pytest
import torch

import oracle
from paper_1204_6367_gb300 import inputs

pytestmark = pytest.mark.gpu
NTH = os.cpu_count() or 1
SHAPES = [dict(block_size=64, hist_per_thread=1, batch_min=1), dict(block_size=128, hist_per_thread=64, batch_min=32),
          dict(block_size=256, hist_per_thread=3, batch_min=3, blocks_per_sm=1),
          dict(block_size=512, hist_per_thread=8, batch_min=20)]


@pytest.fixture(scope="module")
def gd():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1204_6367_gb300 import build, gdrr
    build.build()
    gdrr.lib()
    return gdrr


def _check(gd, prob, n, seed, oopts=None, **opts):
    with gd.Context(prob) as ctx:
        gd.gdrr_set_options(ctx, **opts)
        st = torch.zeros(gd.GDRR_NSTATS, dtype=torch.int64, device="cuda")
        rec = torch.zeros(n * gd.RECORD_DTYPE.itemsize, dtype=torch.uint8, device="cuda")
        p, s = gd.gdrr_mc_project(ctx, n, seed, 0.3, 2, 0, stats=st, records=rec)
        gd.gdrr_sync(ctx)
        got, rec = gd.stats_dict(st), gd.records_array(rec)
    op, os_, ost, orec = oracle.mc_run(prob, n, seed=seed, phi=0.3, angle_index=2, threads=NTH, records=True,
                                       **(oopts or {}))
    assert got == ost
    for f in oracle.RECORD_DTYPE.names:
        np.testing.assert_array_equal(rec[f], orec[f], err_msg=f)
    np.testing.assert_array_equal(p.cpu().numpy(), op)
    np.testing.assert_array_equal(s.cpu().numpy(), os_)


@pytest.mark.parametrize("shape", SHAPES)
def test_launch_shapes(gd, small, shape):
    _check(gd, small, 20_011, 5, **shape)


@pytest.mark.parametrize("shape", SHAPES)
def test_launch_shapes_with_local_majorants(gd, small, shape):
    _check(gd, small, 20_011, 7, oopts=dict(local_majorant=True, cell_shift=2), local_majorant=1, cell_shift=2, **shape)


@pytest.mark.parametrize("block", [256, 512])
def test_eight_materials(gd, block):
    mats = [inputs.AIR, inputs.WATER, inputs.BONE, inputs.LUNG, inputs.ALUMINIUM, inputs.WATER, inputs.BONE, inputs.LUNG]
    prob = inputs.uniform_slab_problem(nx=12, ny=12, nz=12, nu=24, nv=24, det_px=3.0, pencil=False, materials=mats)
    rng = np.random.default_rng(21)
    prob.material[:] = rng.integers(0, 8, prob.material.shape).astype(np.uint8)
    prob.density[:] = rng.uniform(0.1, 2.0, prob.density.shape).astype(np.float32)
    prob.form_factor = None
    _check(gd, prob, 30_000, 3, block_size=block)
