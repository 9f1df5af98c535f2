"""Staged axion-U(1) launches on sizes that their 32-site tiles do not divide, against the gather
launches on the same state: the same equations, the plaquettes' sines and cosines from one sincos
of half the angle instead of the whole, so 2e-6 (FP32) and 1e-13 (FP64) as for the sizes that the
tiles divide; and the Gauss diagnostic, whose maxima and sums do not depend on the form."""
import numpy as np
import pytest

from tests import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def cl():
    from paper_2607_24978_gb300 import build_ext, cl as clmod
    build_ext.build()
    clmod.lib()
    return clmod


FIELDS = ["PHI0", "PI0", "THETA1", "THETA2", "THETA3", "E1", "E2", "E3"]


def run(cl, N, prec, integ, variant, dz, steps=2):
    dtype = np.float64 if prec == 0 else np.float32
    phi, pi = inputs.scalar_state(N, 1, seed=N, fbar=(0.8,), amp=0.2, pamp=0.2)
    th, E = inputs.gauge_state(N, seed=N + 1, theta_amp=0.3, e_amp=0.3)
    with cl.Lattice(N, 0.75 * N, 1, prec, integ, gauge=cl.CL_GAUGE_U1_AXION, expansion=True, alpha=0.5, kappa=0.7,
                    dt=0.01) as g:
        g.cl_set_potential(cl.CL_POT_POLY, [0.8, 0.3, 0.0, 0.0, 0.0])
        g.cl_set_gauge_coupling(2.0, 0.6)
        if variant is not None:
            g.cl_set_option(cl.CL_OPT_PASS_VARIANT, variant)
        if dz:
            g.cl_set_option(cl.CL_OPT_TILE_DZ, dz)
        used = g.cl_get_option(cl.CL_OPT_PASS_VARIANT)
        for name, f in zip(FIELDS, [phi[0], pi[0], *th, *E]):
            g.cl_set_state(getattr(cl, "CL_FIELD_" + name), f.astype(dtype))
        g.cl_set_scalars(1.0, 0.3, 0.0)
        g.cl_step(steps)
        e = g.cl_energies()
        return used, [g.cl_get_state(getattr(cl, "CL_FIELD_" + name)) for name in FIELDS], e


# the narrowest ragged tile (one 16-byte unit), tiles of half a width, last rows of 1 and more,
# chunks of one plane and ragged ones
@pytest.mark.parametrize("N,prec", [(34, 0), (36, 2), (36, 0), (40, 2), (46, 0), (48, 2), (60, 2), (100, 2)])
@pytest.mark.parametrize("integ", ["CL_INT_RK3_3", "CL_INT_VV2"])
@pytest.mark.parametrize("dz", [0, 1, 7])
def test_staged_equals_gather(cl, N, prec, integ, dz):
    if N == 100 and dz == 1:
        pytest.skip("many blocks, covered by the smaller sizes")
    v2, a, ea = run(cl, N, prec, getattr(cl, integ), 2, dz)
    v0, b, eb = run(cl, N, prec, getattr(cl, integ), 0, 0)
    assert (v2, v0) == (2, 0)
    tol = 1e-13 if prec == 0 else 2e-6
    for name, x, y in zip(FIELDS, a, b):
        d = np.linalg.norm((x - y).astype(np.float64)) / np.linalg.norm(y.astype(np.float64))
        assert d < tol, name
    for k in ("a", "adot", "rho", "KE", "GB", "gauss_rms_step", "gauss_violation"):
        assert ea[k] == pytest.approx(eb[k], rel=max(20 * tol, 1e-11)), k


def test_the_librarys_choice(cl):
    for N, prec, want in ((32, 2, 2), (34, 2, 0), (34, 0, 0), (36, 2, 2), (38, 2, 0), (38, 0, 2), (39, 0, 0), (44, 2, 2)):
        with cl.Lattice(N, 10.0, 1, prec, cl.CL_INT_RK3_3, gauge=cl.CL_GAUGE_U1_AXION, kappa=0.7, dt=0.01) as g:
            assert g.cl_get_option(cl.CL_OPT_PASS_VARIANT) == want, (N, prec)
