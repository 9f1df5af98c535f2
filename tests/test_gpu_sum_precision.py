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
