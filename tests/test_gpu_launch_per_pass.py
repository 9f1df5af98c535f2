"""Leapfrog steps of single scalar lattices by a launch per pass.  Small lattices take theirs in
resident launches unless a tiling option is set, as it is in every per-pass arm here; so their sizes
also compare the two where a lattice changes from one to the other."""
import numpy as np
import pytest

from oracle import oracle as O
from tests import inputs
from tests.test_gpu_persist import check, run

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def cl():
    from paper_2607_24978_gb300 import build_ext, cl as mod
    build_ext.build()
    mod.lib()
    return mod


# rows of whole vectors and of any alignment; one and three passes a step (odd: two graphs)
@pytest.mark.parametrize("N", [16, 33])
@pytest.mark.parametrize("integ", ["CL_INT_VV2", "CL_INT_YOSHIDA4"])
@pytest.mark.parametrize("prec", [0, 1, 2])
def test_graphs_and_plain_launches_are_identical(cl, N, integ, prec):
    phi, pi = inputs.scalar_state(N, 1, seed=8, fbar=(1.0,), amp=0.1, pamp=0.1)
    dtype = np.float64 if prec == 0 else np.float32
    outs = []
    for graph in (1, 0):
        with cl.Lattice(N, 5.0, 1, prec, getattr(cl, integ), expansion=True, alpha=0.3, kappa=0.2, dt=0.01) as g:
            g.cl_set_potential(cl.CL_POT_LPHI4, [1.0])
            g.cl_set_option(cl.CL_OPT_GRAPH, graph)
            g.cl_set_option(cl.CL_OPT_TILE_BY, g.cl_get_option(cl.CL_OPT_TILE_BY))
            g.cl_set_state(cl.CL_FIELD_PHI0, phi[0].astype(dtype))
            g.cl_set_state(cl.CL_FIELD_PI0, pi[0].astype(dtype))
            g.cl_set_scalars(1.0)
            for n in (1, 7, 6):
                g.cl_step(n)
            outs.append((g.cl_energies(), g.cl_get_state(cl.CL_FIELD_PHI0), g.cl_get_state(cl.CL_FIELD_PI0)))
    assert outs[0][0] == outs[1][0]
    assert np.array_equal(outs[0][1], outs[1][1]) and np.array_equal(outs[0][2], outs[1][2])


@pytest.mark.parametrize("N", [16, 30, 33])
@pytest.mark.parametrize("prec,tol", [(0, 1e-10), (1, 1e-4), (2, 1e-4)])  # as the library's choice is held to
def test_the_librarys_tiling_matches_the_oracle(cl, N, prec, tol):
    phi, pi = inputs.scalar_state(N, 2, seed=23, fbar=(0.8, 0.1), amp=0.05, pamp=0.05)
    m = O.make_model(N, 0.4 * N, nf=2, alpha=1.0, kappa=0.5, expansion=True, m2=(0.3, 0.2), lam=(1.0, 0.5), g2=2.0)
    st = O.State(phi.copy(), pi.copy(), np.array([1.0, 0.2, 0.0]))
    with cl.Lattice(N, 0.4 * N, 2, prec, cl.CL_INT_YOSHIDA4, expansion=True, alpha=1.0, kappa=0.5, dt=0.02) as g:
        g.cl_set_potential(cl.CL_POT_POLY, [0.3, 1.0, 0.2, 0.5, 2.0])
        g.cl_set_option(cl.CL_OPT_TILE_BY, g.cl_get_option(cl.CL_OPT_TILE_BY))
        for f in range(2):
            g.cl_set_state(cl.CL_FIELD_PHI0 + f, phi[f].astype(g.dtype))
            g.cl_set_state(cl.CL_FIELD_PI0 + f, pi[f].astype(g.dtype))
        g.cl_set_scalars(*st.abt)
        g.cl_step(12)
        e = g.cl_energies()
        got = [g.cl_get_state(f) for f in (cl.CL_FIELD_PHI0, cl.CL_FIELD_PHI1, cl.CL_FIELD_PI0, cl.CL_FIELD_PI1)]
    O.step(m, st, O.YOSHIDA4, 0.02, 12)
    for x, y in zip(got, list(st.phi) + list(st.pi)):
        assert np.linalg.norm((x - y).ravel()) <= tol * np.linalg.norm(y.ravel())
    assert e["a"] == pytest.approx(st.abt[0], rel=tol) and e["step"] == 12


# the largest lattices that the resident launches take, and the next ones, of each kind: many rounds
# of the threads over a box, ragged boxes, every SM
@pytest.mark.parametrize("N,nf,prec", [(100, 1, 0), (101, 1, 0), (73, 2, 0), (74, 2, 0), (128, 1, 1), (132, 1, 1),
                                       (120, 2, 1), (124, 2, 1), (131, 2, 1), (133, 1, 1), (144, 1, 2), (132, 2, 2)])
def test_resident_launches_at_their_largest_sizes(cl, N, nf, prec):
    a, b = (run(cl, N, nf, prec, cl.CL_INT_YOSHIDA4, (2, 1), r) for r in (True, False))
    check(a, b, prec)


# calls of one and of a few passes on lattices that take longer ones in resident launches: the same
# bits as with a tiling option set, where the call launches every pass
@pytest.mark.parametrize("N,nf,prec,passes", [(41, 1, 1, 1), (64, 2, 1, 1), (96, 1, 0, 1), (100, 2, 1, 2), (125, 1, 1, 2)])
def test_calls_of_few_passes_are_launched_one_by_one(cl, N, nf, prec, passes):
    phi, pi = inputs.scalar_state(N, nf, seed=5, fbar=(1.0, 0.1), amp=0.05, pamp=0.05)
    dtype = np.float64 if prec == 0 else np.float32
    outs = []
    for tiled, calls in ((False, [passes] * 4), (True, [passes] * 4), (False, [4 * passes])):
        with cl.Lattice(N, 0.4 * N, nf, prec, cl.CL_INT_VV2, expansion=True, alpha=0.3, kappa=0.2, dt=0.01) as g:
            g.cl_set_potential(cl.CL_POT_POLY, [0.5, 1.0] + ([0.2, 0.4, 3.0] if nf == 2 else [0.0] * 3))
            if tiled:
                g.cl_set_option(cl.CL_OPT_TILE_BY, g.cl_get_option(cl.CL_OPT_TILE_BY))
            for f in range(nf):
                g.cl_set_state(cl.CL_FIELD_PHI0 + f, phi[f].astype(dtype))
                g.cl_set_state(cl.CL_FIELD_PI0 + f, pi[f].astype(dtype))
            g.cl_set_scalars(1.0)
            for n in calls:
                g.cl_step(n)
            outs.append(g.cl_energies())
    assert outs[0] == outs[1]
    for k in ("a", "adot", "rho"):
        assert outs[0][k] == pytest.approx(outs[2][k], rel=1e-7 if prec else 1e-11)
    assert outs[0] != outs[2]  # the longer call is a resident one: its sums have another order
