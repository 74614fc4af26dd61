"""reconstruct takes views of the context's detector and refuses other shapes,
also those of the same size (no GPU: the kernels' calls are stood in for)."""
import types

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1204_6367_gb300 import gdrr, scan  # noqa: E402

NV, NU = 3, 5


@pytest.fixture()
def ctx(monkeypatch):
    monkeypatch.setattr(gdrr, "gdrr_air_scan", lambda c: torch.ones((NV, NU), dtype=torch.float64))
    monkeypatch.setattr(gdrr, "gdrr_line_integrals_views", lambda s, a, floor: s.float())
    monkeypatch.setattr(gdrr, "fdk", lambda geo, g, angles: g)
    prob = types.SimpleNamespace(sad=900.0, sdd=1400.0, du=1.0, dv=1.0)
    return types.SimpleNamespace(prob=prob, nu=NU, nv=NV)


def test_views_of_the_detector(ctx):
    sig = torch.ones((4, NV, NU), dtype=torch.float64)
    assert scan.reconstruct(ctx, np.zeros(4), sig, (2, 2, 2), (1.0, 1.0, 1.0)).shape == sig.shape


@pytest.mark.parametrize("shape", [(4, NU, NV), (4, NV * NU), (4, NV * NU, 1), (4 * NV * NU,), (4, 1, NU), (4, NV, NU, 1)])
def test_other_shapes_are_refused(ctx, shape):
    with pytest.raises((RuntimeError, ValueError)):
        scan.reconstruct(ctx, np.zeros(4), torch.ones(shape, dtype=torch.float64), (2, 2, 2), (1.0, 1.0, 1.0))
