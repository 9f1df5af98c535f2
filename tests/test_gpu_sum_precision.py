"""Lattice sums keep the bits that the terms have: terms of very different size, chosen so that the
sum is exact in FP64 (or in compensated FP32) and not in a shorter accumulator.

With dt = 1e-30 the kicks round away and pi stays what was uploaded; K0 = sum pi^2 / (2 a^6 N^3)
with a = 1 has no rounding of its own where N^3 is a power of two."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def cl():
    from paper_2607_24978_gb300 import build_ext, cl as mod
    build_ext.build()
    mod.lib()
    return mod


def kinetic(cl, N, prec, values, options=()):
    """K0 of the last of three passes over a lattice with pi = values[(z, y, x)], 0 elsewhere."""
    pi = np.zeros((N, N, N), np.float32)
    for at, v in values.items():
        pi[at] = v
    with cl.Lattice(N, 1.0 * N, 1, prec, cl.CL_INT_VV2, expansion=False, dt=1e-30) as g:
        g.cl_set_potential(cl.CL_POT_LPHI4, [1.0])
        for o, v in options:
            g.cl_set_option(o, v)
        g.cl_set_state(cl.CL_FIELD_PHI0, np.zeros_like(pi))
        g.cl_set_state(cl.CL_FIELD_PI0, pi)
        g.cl_set_scalars(1.0)
        g.cl_step(3)
        K0 = g.cl_energies()["K0"]
        assert np.array_equal(g.cl_get_state(cl.CL_FIELD_PI0), pi)
    return K0


@pytest.mark.parametrize("prec", [1, 2])
def test_resident_launches_add_warps_in_fp64(cl, prec):
    """Three rows of one block's box, a warp each at N = 32: 2^26 + 1 + 2^-26 fills FP64's 53 bits
    (a pair of floats holds 2^26 and 1 and loses the rest)."""
    K0 = kinetic(cl, 32, prec, {(0, 0, 0): 2.0**13, (0, 1, 0): 1.0, (0, 2, 0): 2.0**-13})
    assert K0 == (2.0**26 + 1.0 + 2.0**-26) / 2.0**16


# sites of one thread: 0, 32, 64 and 96 along the tile's rows (N = 33: x = 0 and 32 of row 0, 31 of
# row 1, 30 of row 2)
@pytest.mark.parametrize("small", [(0, 0, 32), (0, 1, 31), (0, 2, 30)])
@pytest.mark.parametrize("prec", [1, 2])
def test_rows_of_any_alignment_add_every_site_compensated(cl, prec, small):
    """1 + 2^-26 needs 27 bits, more than FP32 has: lost (1.5e-8 relative) where two sites are added
    before the compensated sum, kept to 1e-14 where each is added to it."""
    N = 33
    K0 = kinetic(cl, N, prec, {(0, 0, 0): 1.0, small: 2.0**-13}, ((cl.CL_OPT_STAGES, 4),))
    assert K0 == pytest.approx((1.0 + 2.0**-26) / (2.0 * N**3), rel=1e-12, abs=0.0)


# the gather launches, and the staged ones on a size that is no multiple of their 32-column tiles
@pytest.mark.parametrize("N", [16, 36])
@pytest.mark.parametrize("integ", ["CL_INT_RK3_3", "CL_INT_VV2"])
def test_gauss_tracking_of_weak_fields(cl, N, integ):
    """E = 2^-60 but for one link, a unit in the last place (2^-83) larger: the charge is 2^-83 on two
    sites, its square 2^-166 below FP32's range, E^2 = 2^-120 within it."""
    E = np.full((N, N, N), 2.0**-60, np.float32)
    E[3, 5, 7] = np.float32(2.0**-60 * (1.0 + 2.0**-23))
    zero = np.zeros_like(E)
    with cl.Lattice(N, 1.0 * N, 1, cl.CL_PREC_FP32, getattr(cl, integ), gauge=cl.CL_GAUGE_U1_AXION, expansion=False,
                    alpha=1.0, dt=1e-6) as g:
        g.cl_set_potential(cl.CL_POT_LPHI4, [1.0])
        g.cl_set_gauge_coupling(1.0, 1.0)
        for f in (cl.CL_FIELD_PHI0, cl.CL_FIELD_PI0):
            g.cl_set_state(f, zero)
        for i in range(3):
            g.cl_set_state(cl.CL_FIELD_THETA1 + i, zero)
            g.cl_set_state(cl.CL_FIELD_E1 + i, E if i == 0 else zero)
        g.cl_set_scalars(1.0)
        g.cl_step(1)
        r = g.cl_energies()["gauss_rms_step"]
    assert r == pytest.approx(2.0**0.5 * 2.0**-23 / N**1.5, rel=1e-6, abs=0.0)
