"""Staged axion-U(1) launches with tiles of other widths than 32 columns (whole rows, several rows a
warp, idle warps, tiles that end inside and outside the lattice), against the gather launches on the
same state; bounds as for the other staged sizes, 2e-6 (FP32) and 1e-13 (FP64)."""
import numpy as np
import pytest

from tests.test_gpu_u1_ragged import FIELDS, cl, run  # noqa: F401 (cl is the fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,prec", [(44, 2), (52, 2), (68, 2), (132, 2), (38, 0), (90, 0)])
@pytest.mark.parametrize("integ", ["CL_INT_RK3_3", "CL_INT_VV2"])
def test_tiles_equal_gather(cl, N, prec, integ):
    v2, a, _ = run(cl, N, prec, getattr(cl, integ), None, 0)
    v0, b, _ = run(cl, N, prec, getattr(cl, integ), 0, 0)
    assert (v2, v0) == (2, 0)
    tol = 1e-13 if prec == 0 else 2e-6
    for name, x, y in zip(FIELDS, a, b):
        d = np.linalg.norm((x - y).astype(np.float64)) / np.linalg.norm(y.astype(np.float64))
        assert d < tol, name
