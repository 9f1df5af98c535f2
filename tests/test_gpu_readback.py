"""Reads of an open leapfrog share one synchronising pass: what is read, and what a read reports,
must be as if each read closed the leapfrog anew."""
import numpy as np
import pytest

from tests import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def cl():
    from paper_2607_24978_gb300 import build_ext, cl as mod
    build_ext.build()
    mod.lib()
    return mod


def lattice(cl, N=24, **kw):
    g = cl.Lattice(N, 9.0, 2, cl.CL_PREC_FP32_KAHAN, cl.CL_INT_YOSHIDA4, expansion=True, alpha=1.0, kappa=0.2, dt=0.01, **kw)
    g.cl_set_potential(cl.CL_POT_M2_G2, [1.0, 3.0])
    phi, pi = inputs.scalar_state(N, 2, seed=4, fbar=(1.0, 0.1), amp=0.05, pamp=0.05)
    for f in range(2):
        g.cl_set_state(cl.CL_FIELD_PHI0 + f, phi[f].astype(np.float32))
        g.cl_set_state(cl.CL_FIELD_PI0 + f, pi[f].astype(np.float32))
    g.cl_set_scalars(1.0)
    return g


READS = [lambda cl, g: g.cl_get_state(cl.CL_FIELD_PI0), lambda cl, g: g.cl_get_state(cl.CL_FIELD_PI1),
         lambda cl, g: g.cl_get_state(cl.CL_FIELD_PHI1), lambda cl, g: np.array(g.cl_get_scalars()),
         lambda cl, g: g.cl_spectrum(cl.CL_FIELD_PI1)[2], lambda cl, g: np.array([g.cl_energies()["rho"]])]
# what may come between two reads: nothing, a step, a change of the potential (the closing kick
# changes with it) or of the tiling, an upload (closes and reopens), a trial pass of the autotuner
BETWEEN = {"nothing": lambda cl, g: None, "step": lambda cl, g: g.cl_step(1),
           "potential": lambda cl, g: g.cl_set_potential(cl.CL_POT_M2_G2, [2.0, 5.0]),
           "tiling": lambda cl, g: g.cl_set_option(cl.CL_OPT_TILE_BY, 3),
           "upload": lambda cl, g: (g.cl_set_state(cl.CL_FIELD_PI0, np.full((24,) * 3, 0.25, np.float32)), g.cl_step(1)),
           "autotune": lambda cl, g: g.cl_autotune()}


@pytest.mark.parametrize("between", sorted(BETWEEN))
def test_repeated_reads_equal_first_reads(cl, between):
    def run(prior):  # the reads after `between`, with or without all of them before it
        with lattice(cl) as g:
            g.cl_step(3)
            if prior:
                for r in READS:
                    r(cl, g)
            BETWEEN[between](cl, g)
            return [r(cl, g) for r in READS] + [r(cl, g) for r in READS]

    first, again = run(False), run(True)
    for k, (a, b) in enumerate(zip(first, again)):
        if between == "autotune":  # its choice of tiling may differ: sums in another order
            assert np.allclose(a, b, rtol=1e-5, atol=1e-6), k
        else:
            assert np.array_equal(a, b), k
    n = len(READS)
    for k in range(n):
        assert np.array_equal(first[k], first[n + k]), k


def test_ensemble_members_read_in_any_order(cl):
    sizes = [8, 12, 16]
    with cl.Lattice(8, 5.0, 1, cl.CL_PREC_FP32_KAHAN, cl.CL_INT_VV2, alpha=1.0, kappa=0.2, dt=0.01, member_N=sizes) as g:
        g.cl_set_potential(cl.CL_POT_LPHI4, [1.0])
        g.cl_init_vacuum(5, 1e30, 1e-3, (1.0,))
        g.cl_step(3)
        a = [g.cl_get_state(cl.CL_FIELD_PI0, member=m) for m in range(3)]
        b = [g.cl_get_state(cl.CL_FIELD_PI0, member=m) for m in (2, 0, 1)]
        for x, y in zip(a, (b[1], b[2], b[0])):
            assert np.array_equal(x, y)
        g.cl_step(1)
        assert not np.array_equal(a[1], g.cl_get_state(cl.CL_FIELD_PI0, member=1))


def test_every_read_reports_a_violated_limit(cl):
    with lattice(cl) as g:
        g.cl_step(2)
        g.cl_get_state(cl.CL_FIELD_PI0)
        g.cl_set_hubble_limit(1e-30)
        for f in (cl.CL_FIELD_PI0, cl.CL_FIELD_PI1, cl.CL_FIELD_PI0):
            with pytest.raises(cl.CLError) as e:
                g.cl_get_state(f)
            assert e.value.status == cl.CL_ECONSTRAINT
        g.cl_set_hubble_limit(0.0)
        g.cl_get_state(cl.CL_FIELD_PI0)
