"""Steps of small lattices in resident multi-pass launches (the library's choice) against one
launch per pass (chosen by setting a tiling option).

The sites' rounded operations are the same in FP32; a(t) differs by FP64 rounding of sums taken
in another order (1e-16 relative in FP64 fields, whose gradient sum also takes another form;
1e-12 in the compensated FP32 sums), which moves an FP32 drift factor by an ulp (6e-8) only in
rare ties.  FP32 fields therefore agree to 1e-6 over these runs, FP64 ones to 1e-12."""
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


def run(cl, N, nf, prec, integ, calls, resident, expansion=True, alpha=0.5, dt=0.005, limit=0.0, nan=False):
    phi, pi = inputs.scalar_state(N, nf, seed=N + nf, fbar=(1.0, 0.1), amp=0.05, pamp=0.05)
    dtype = np.float64 if prec == 0 else np.float32
    with cl.Lattice(N, 0.4 * N, nf, prec, integ, expansion=expansion, alpha=alpha, kappa=0.2, dt=dt) as g:
        g.cl_set_potential(cl.CL_POT_POLY, [0.5, 1.0, 0.2 if nf == 2 else 0.0, 0.4 if nf == 2 else 0.0,
                                            3.0 if nf == 2 else 0.0])
        if not resident:
            g.cl_set_option(cl.CL_OPT_TILE_BY, max(1, min(N, 128 // N)))
        if limit:
            g.cl_set_hubble_limit(limit)
        for f in range(nf):
            if nan:
                phi[f][0, 0, 0] = np.nan
            g.cl_set_state(cl.CL_FIELD_PHI0 + f, phi[f].astype(dtype))
            g.cl_set_state(cl.CL_FIELD_PI0 + f, pi[f].astype(dtype))
        g.cl_set_scalars(1.0, 0.3, 0.0)
        launches = []
        for n in calls:
            g.cl_step(n)
            launches.append(g.cl_last_launch_count())
        e = g.cl_energies()  # the last pass's, before a read closes the leapfrog
        fields = [g.cl_get_state(f) for f in list(range(nf)) + [cl.CL_FIELD_PI0 + f for f in range(nf)]]
        return fields, e, launches, g.cl_get_scalars()


def check(a, b, prec):
    tol = 1e-12 if prec == 0 else 1e-6
    for x, y in zip(a[0], b[0]):
        assert np.max(np.abs(x - y)) <= tol * np.max(np.abs(y))
    etol = 1e-11 if prec == 0 else 1e-7
    for k in ("t", "a", "adot", "K0", "K1", "G0", "G1", "V", "rho", "p"):
        assert a[1][k] == pytest.approx(b[1][k], rel=etol, abs=1e-300), k
    assert a[1]["step"] == b[1]["step"] and a[2] == b[2]
    assert a[3] == pytest.approx(b[3], rel=etol)


# sizes: two and three sites a row (all neighbours coincide), a part of a warp, boxes with ragged
# rows and planes, one and several rounds of the threads, more blocks than half the SMs
@pytest.mark.parametrize("N", [2, 3, 8, 17, 32, 33, 48, 70])
@pytest.mark.parametrize("nf,prec", [(1, 1), (2, 1), (1, 2), (2, 2), (1, 0), (2, 0)])
def test_resident_launches_equal_a_launch_per_pass(cl, N, nf, prec):
    a, b = (run(cl, N, nf, prec, cl.CL_INT_YOSHIDA4, (3, 1), r) for r in (True, False))
    check(a, b, prec)


@pytest.mark.parametrize("integ,calls", [("CL_INT_VV2", (2500, 3)), ("CL_INT_YOSHIDA10", (2, 30)), ("CL_INT_YOSHIDA6", (1, 4))])
def test_schedules_and_runs_longer_than_a_launch(cl, integ, calls):
    """81 passes a step; calls of more passes than one launch takes, of odd and even counts."""
    a, b = (run(cl, 9, 1, 0, getattr(cl, integ), calls, r, dt=0.001) for r in (True, False))
    check(a, b, 0)


@pytest.mark.parametrize("expansion,alpha", [(False, 1.0), (True, 0.0), (True, 1.0), (True, 0.3)])
def test_backgrounds(cl, expansion, alpha):
    for prec in (0, 1):
        a, b = (run(cl, 20, 2, prec, cl.CL_INT_VV2, (5,), r, expansion=expansion, alpha=alpha) for r in (True, False))
        check(a, b, prec)


def test_status_is_reported(cl):
    for kw, status in ((dict(nan=True), cl.CL_ENAN), (dict(limit=1e-30), cl.CL_ECONSTRAINT),
                       (dict(nan=True, expansion=False), cl.CL_ENAN)):
        with pytest.raises(cl.CLError) as e:
            run(cl, 16, 1, 1, cl.CL_INT_VV2, (4,), True, **kw)
        assert e.value.status == status
