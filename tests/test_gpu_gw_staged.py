"""The staged GW pass (one component a work unit) against the direct one (CL_OPT_STAGES -1) on the
same state.  The source's (1/2dx)^2 is folded into its prefactor and the trace of the diagonal
components is subtracted in another order, a few FP32 roundings of each kick: 2e-6 relative to the
largest value after a few steps."""
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


# last tiles of few rows, rows of less than a warp and of several; units in one wave and in many
@pytest.mark.parametrize("N,nf,prec,integ", [(96, 1, 1, "CL_INT_VV2"), (96, 2, 2, "CL_INT_YOSHIDA4"), (100, 2, 1, "CL_INT_VV2"),
                                             (108, 1, 2, "CL_INT_VV2"), (132, 2, 1, "CL_INT_VV2"), (256, 2, 1, "CL_INT_VV2")])
def test_staged_equals_direct(cl, N, nf, prec, integ):
    phi, pi = inputs.scalar_state(N, nf, seed=N, fbar=(1.0, 0.1), amp=0.05, pamp=0.05)
    g0 = inputs.rng(N + 1)
    v = 1e-3 * g0.standard_normal((10, N, N, N)).astype(np.float32)
    outs = []
    for stages in (-1, 0):
        with cl.Lattice(N, 0.4 * N, nf, prec, getattr(cl, integ), expansion=True, alpha=0.5, kappa=0.2, dt=0.01) as g:
            g.cl_set_potential(cl.CL_POT_POLY, [0.5, 1.0, 0.2 if nf == 2 else 0.0, 0.0, 3.0 if nf == 2 else 0.0])
            g.cl_enable_gw()
            g.cl_set_option(cl.CL_OPT_STAGES, stages)
            for f in range(nf):
                g.cl_set_state(cl.CL_FIELD_PHI0 + f, phi[f].astype(np.float32))
                g.cl_set_state(cl.CL_FIELD_PI0 + f, pi[f].astype(np.float32))
            for q in range(10):
                g.cl_set_state(cl.CL_FIELD_GW_V11 + q, v[q])
            g.cl_set_scalars(1.0, 0.3, 0.0)
            g.cl_step(2)
            outs.append([g.cl_get_state(cl.CL_FIELD_GW_V11 + q) for q in range(10)])
    for q, (a, b) in enumerate(zip(*outs)):
        assert np.max(np.abs(a - b)) <= 2e-6 * np.max(np.abs(b)), q
