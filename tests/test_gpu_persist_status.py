"""What the resident launches of a small lattice report of their own passes: the opening half-kick is
an ordinary pass, so every condition here arises after it (cl_sync has found nothing wrong).

A Hubble limit makes block 0 add up every pass's energies beside the passes that follow; the largest
violation that the per-pass kernel reports over the same steps must be met by a limit just above it
and break one just below it.  FP64 sums agree to 1e-13 relative between the two forms and the
violation is 1e-5 to 1e-2 of the terms whose difference it is, hence to 1e-8; the bounds leave a
factor of 10.  FP32 fields differ by up to 1e-6 between the two forms over such runs (rare ties of
a drift factor); moving every site of the state by 1e-6 moved the largest violation by 6e-5
relative in the oracle, so 2e-3 is left."""
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


def opened(cl, N, prec, alpha, resident=True, amp=0.05, dt=0.05, integ=None, expansion=True, fbar=1.0):
    """A lattice whose leapfrog is open, after one step with a clean status."""
    phi, pi = inputs.scalar_state(N, 1, seed=N, fbar=(fbar,), amp=amp, pamp=amp)
    dtype = np.float64 if prec == 0 else np.float32
    g = cl.Lattice(N, 0.4 * N, 1, prec, cl.CL_INT_VV2 if integ is None else integ, expansion=expansion, alpha=alpha,
                   kappa=0.5, dt=dt)
    g.cl_set_potential(cl.CL_POT_LPHI4, [1.0])
    if not resident:
        g.cl_set_option(cl.CL_OPT_STAGES, -1)
    g.cl_set_state(cl.CL_FIELD_PHI0, phi[0].astype(dtype))
    g.cl_set_state(cl.CL_FIELD_PI0, pi[0].astype(dtype))
    g.cl_set_scalars(1.0)
    g.cl_step(1)
    g.cl_sync()
    return g


@pytest.mark.parametrize("N,passes", [(8, 2500), (32, 2500), (70, 700)])
@pytest.mark.parametrize("alpha", [1.0, 0.3])
@pytest.mark.parametrize("prec", [0, 1])
def test_hubble_limit_that_holds_and_one_that_does_not(cl, N, passes, alpha, prec):
    with opened(cl, N, prec, alpha, resident=False) as g:
        hv = []
        for _ in range(passes):
            g.cl_step(1)
            hv.append(g.cl_energies()["hubble_violation"])
    worst, tol = max(hv), 1e-7 if prec == 0 else 2e-3
    assert 1e-5 < worst < 0.5
    with opened(cl, N, prec, alpha) as g:
        g.cl_set_hubble_limit(worst * (1.0 + tol))
        g.cl_step(passes)
        g.cl_sync()
        assert g.cl_energies()["hubble_violation"] == pytest.approx(hv[-1], rel=tol)
    with opened(cl, N, prec, alpha) as g:
        g.cl_set_hubble_limit(worst * (1.0 - tol))
        g.cl_step(passes)
        with pytest.raises(cl.CLError) as e:
            g.cl_sync()
        assert e.value.status == cl.CL_ECONSTRAINT


@pytest.mark.parametrize("expansion", [True, False])
def test_values_that_overflow_within_a_launch(cl, expansion):
    """phi'' = -phi^3 with steps far beyond the stability limit: FP32 overflows in a few steps."""
    with opened(cl, 16, 1, 1.0, dt=3.0, expansion=expansion, fbar=2.0) as g:
        g.cl_step(60)
        with pytest.raises(cl.CLError) as e:
            g.cl_sync()
        assert e.value.status == cl.CL_ENAN
