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
