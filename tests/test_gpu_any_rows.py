"""The staged scalar pass on FP32 rows that are no multiple of 16 bytes (N % 4 != 0) against the
direct loader (CL_OPT_STAGES -1).

Both apply the same rounded operations to every site, so the fields must agree bit for bit; the
volume averages are sums of the same per-site terms in another order and with another
contraction, each term good to FP32 rounding (2^-24 = 6e-8 relative), so they agree to 1e-7."""
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


# sizes: two sites a row; tiles of one warp, of a part of a warp, of several; rows longer than a
# warp's 128 sites; halo rows that wrap with another shift (odd N) and the same (N % 4 == 2);
# the longest odd row.  by/dz: one row, ragged last tiles and chunks, persistent ranges, the
# library's choice.
@pytest.mark.parametrize("N,by,dz", [(2, 0, 0), (3, 1, 1), (5, 2, 3), (7, 0, -1), (33, 5, 0), (34, 0, 7), (66, 4, -1),
                                     (131, 0, 0), (131, 3, 50), (258, 2, 100)])
@pytest.mark.parametrize("nf,prec", [(1, 1), (2, 1), (2, 2)])
def test_fields_equal_the_direct_loader(cl, N, by, dz, nf, prec):
    phi, pi = inputs.scalar_state(N, nf, seed=N + nf, fbar=(1.0, 0.1), amp=0.05, pamp=0.05)
    outs = []
    for stages in (-1, 3, 4):
        with cl.Lattice(N, 0.3 * N, nf, prec, cl.CL_INT_YOSHIDA4, expansion=True, alpha=0.5, kappa=0.2, dt=0.01) as g:
            g.cl_set_potential(cl.CL_POT_POLY, [0.5, 1.0, 0.2 if nf == 2 else 0.0, 0.4 if nf == 2 else 0.0,
                                                3.0 if nf == 2 else 0.0])
            if by:
                g.cl_set_option(cl.CL_OPT_TILE_BY, by)
            if dz:
                g.cl_set_option(cl.CL_OPT_TILE_DZ, dz)
            g.cl_set_option(cl.CL_OPT_STAGES, stages)
            assert g.cl_get_option(cl.CL_OPT_STAGES) == max(stages, 0)
            for f in range(nf):
                g.cl_set_state(cl.CL_FIELD_PHI0 + f, phi[f].astype(np.float32))
                g.cl_set_state(cl.CL_FIELD_PI0 + f, pi[f].astype(np.float32))
            g.cl_set_scalars(1.0, 0.3, 0.0)
            g.cl_step(1)
            fields = [g.cl_get_state(f) for f in list(range(nf)) + [cl.CL_FIELD_PI0 + f for f in range(nf)]]
            outs.append((fields, g.cl_energies()))
    for fields, e in outs[1:]:
        for a, b in zip(fields, outs[0][0]):
            # one step: a(t) of the two differs by the rounding of the energies only after its
            # first pass, far below half an FP32 ulp of the drift factor but for rare ties
            assert np.mean(a != b) < 1e-3
            assert np.max(np.abs(a - b)) <= 4e-7 * np.max(np.abs(b))
        for k in ("a", "adot", "K0", "G0", "V", "rho"):
            assert e[k] == pytest.approx(outs[0][1][k], rel=1e-7), k


def test_autotune_keeps_the_staged_pass_available(cl):
    """The autotuner's candidates include the staged pass on such rows; the state is unchanged."""
    N = 99
    phi, pi = inputs.scalar_state(N, 1, seed=3, fbar=(1.0,), amp=0.05, pamp=0.05)
    with cl.Lattice(N, 0.3 * N, 1, 1, cl.CL_INT_VV2, expansion=True, alpha=1.0, kappa=0.2, dt=0.01) as g:
        g.cl_set_potential(cl.CL_POT_LPHI4, [1.0])
        g.cl_set_state(cl.CL_FIELD_PHI0, phi[0].astype(np.float32))
        g.cl_set_state(cl.CL_FIELD_PI0, pi[0].astype(np.float32))
        g.cl_set_scalars(1.0)
        stages, by, dz, us, variant = g.cl_autotune()
        assert (stages, by, dz, variant) == tuple(g.cl_get_option(o) for o in (
            cl.CL_OPT_STAGES, cl.CL_OPT_TILE_BY, cl.CL_OPT_TILE_DZ, cl.CL_OPT_PASS_VARIANT))
        assert stages in (3, 4)  # measured 2.0 times the direct loader at this size
        assert np.array_equal(g.cl_get_state(cl.CL_FIELD_PHI0), phi[0].astype(np.float32))
