"""The per-warp photon pool of the transport at the edges of its lists:
launches smaller than a warp, a pool and the grid, ragged multi-job launches,
history ids that carry into their high word, and odd macro-cell grids.  Every
tally and counter equals the CPU oracle's exactly (the transport's arithmetic
is FP32, operation for operation)."""
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


@pytest.fixture(scope="module")
def odd():
    """A ragged phantom (37 x 29 x 23 voxels, outer half voxels filled) of three materials."""
    p = inputs.torso_problem(vox=8.0, nu=40, nv=30, det_px=9.9)
    p.material = np.ascontiguousarray(p.material[:23, 17:46, 13:50])
    p.density = np.ascontiguousarray(p.density[:23, 17:46, 13:50])
    return p


def _check(gd, prob, n, seed, offset=0, angle=0.7, oopts=None, **opts):
    with gd.Context(prob) as ctx:
        gd.gdrr_set_options(ctx, **opts)
        shift = gd.gdrr_get_options(ctx)["cell_shift"]
        st = torch.zeros(gd.GDRR_NSTATS, dtype=torch.int64, device="cuda")
        p, s = gd.gdrr_mc_project(ctx, n, seed, angle, 3, offset, stats=st)
        gd.gdrr_sync(ctx)
        got = gd.stats_dict(st)
        skips = gd.cell_skips(st)
    op, os_, ost, _ = oracle.mc_run(prob, n, seed=seed, phi=angle, angle_index=3, history_offset=offset, threads=NTH,
                                    cell_shift=max(shift, 1), **(oopts or {}))
    assert got == ost
    np.testing.assert_array_equal(p.cpu().numpy(), op)
    np.testing.assert_array_equal(s.cpu().numpy(), os_)
    return got, skips


@pytest.mark.parametrize("pool", [-1, 1, 3])
@pytest.mark.parametrize("n", [1, 31, 33, 97, 3649, 30_011])
def test_small_launches(gd, odd, n, pool):
    _check(gd, odd, n, 5, photon_pool=pool)


@pytest.mark.parametrize("shift", [-1, 1, 2, 6])
def test_cells_of_a_ragged_phantom(gd, odd, shift):
    got, skips = _check(gd, odd, 40_000, 6, cell_shift=shift)
    assert (skips == 0) if shift < 0 else (0 < skips < got["virtual"])


@pytest.mark.parametrize("kind", ["local", "form-factor", "nearest", "filter", "local-ff"])
def test_options_at_odd_sizes(gd, odd, kind):
    o = {"local": dict(local_majorant=1), "form-factor": dict(rayleigh_form_factor=1), "nearest": dict(nearest_voxel=1),
         "filter": dict(scatter_filter=3), "local-ff": dict(local_majorant=1, rayleigh_form_factor=1)}[kind]
    names = {"rayleigh_form_factor": "rayleigh_ff"}
    for n in (33, 20_011):
        _check(gd, odd, n, 7, oopts={names.get(k, k): (bool(v) if k != "scatter_filter" else v) for k, v in o.items()}, **o)


def test_history_ids_carry(gd, odd):
    _check(gd, odd, 20_000, 8, offset=(1 << 32) - 9_001)


def test_two_materials_and_step_limit(gd):
    p = inputs.uniform_slab_problem(nx=15, ny=9, nz=11, materials=[inputs.AIR, inputs.WATER], pencil=False)
    _check(gd, p, 20_011, 9, angle=0.3)
    _check(gd, p, 5_003, 9, angle=0.3, oopts=dict(max_steps=3), max_steps=3)


def test_ragged_jobs_equal_single_calls(gd, odd):
    angles, budgets = np.array([0.0, 1.1, 2.9, 4.0]), np.array([7, 20_003, 0, 311], np.uint64)
    with gd.Context(odd) as ctx:
        bp, bs = gd.gdrr_mc_project_batched(ctx, angles, budgets, 4)
        for a in range(4):
            p, s = gd.gdrr_mc_project(ctx, int(budgets[a]), 4, float(angles[a]), a)
            assert torch.equal(p, bp[a]) and torch.equal(s, bs[a])


@pytest.mark.parametrize("shift", [4, 5, 6])
@pytest.mark.parametrize("extra", [{}, {"rayleigh_form_factor": 1}, {"max_steps": 9}])
def test_local_majorants_in_coarse_cells(gd, odd, shift, extra):
    names = {"rayleigh_form_factor": "rayleigh_ff"}
    oopts = {names.get(k, k): (True if k == "rayleigh_form_factor" else v) for k, v in extra.items()}
    _check(gd, odd, 20_011, 9, oopts={"local_majorant": True, **oopts}, local_majorant=1, cell_shift=shift, **extra)
