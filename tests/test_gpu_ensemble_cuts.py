"""The library's cuts of an ensemble into blocks of equal work against whole columns, and the
members' status words read together.

Cutting a column moves no field value; it reorders the FP64 sums of a and a', so the fields agree
to a few rounding errors a step (bound 1e-13 in FP64, as between other work-item shapes)."""
import numpy as np
import pytest

from tests import inputs
from tests.test_gpu_ensemble import member_params, rel_l2, run_ensemble

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def cl():
    from paper_2607_24978_gb300 import build_ext, cl as mod
    build_ext.build()
    mod.lib()
    return mod


# shorter than an item's least planes; parts of a column of every length; two blocks' worth of a
# large member beside small ones; more columns than a wave of blocks; rows of any alignment
@pytest.mark.parametrize("sizes", [[7, 3, 2], [33, 16, 9], [96, 8], [16] * 700, [35, 27, 10] * 5])
@pytest.mark.parametrize("nf", [1, 2])
def test_cut_columns_equal_whole_columns(cl, sizes, nf):
    base = {n: member_params([n], nf, seed=n)[0] for n in set(sizes)}
    params = [base[n] for n in sizes]
    a = run_ensemble(cl, params, nf, 0, 1, 0.02, 3)
    b = run_ensemble(cl, params, nf, 0, 1, 0.02, 3, opts=((cl.CL_OPT_TILE_DZ, max(sizes)),))
    for m in range(len(sizes)):
        assert rel_l2(a[0][m], b[0][m]) < 1e-13, m
        assert rel_l2(a[1][m], b[1][m]) < 1e-13, m
        assert a[2][m]["a"] == pytest.approx(b[2][m]["a"], rel=1e-14)


@pytest.mark.parametrize("members,bad", [(3, 1), (40, 39), (1100, 1050)])
def test_any_members_status_is_reported_once(cl, members, bad):
    with cl.Lattice(4, 3.0, 1, cl.CL_PREC_FP64, cl.CL_INT_VV2, alpha=1.0, kappa=0.2, dt=0.01, member_N=[4] * members) as g:
        g.cl_set_potential(cl.CL_POT_LPHI4, [1.0])
        phi, pi = inputs.scalar_state(4, 1, seed=4)
        for m in range(members):
            g.cl_set_state(cl.CL_FIELD_PHI0, phi[0] if m != bad else np.full((4, 4, 4), 1e200), member=m)
            g.cl_set_state(cl.CL_FIELD_PI0, pi[0], member=m)
        g.cl_set_scalars(1.0, 0.0, 0.0)
        g.cl_step(1)
        with pytest.raises(cl.CLError) as e:
            g.cl_get_state(cl.CL_FIELD_PHI0, member=0)
        assert e.value.status == cl.CL_ENAN
        g.cl_get_state(cl.CL_FIELD_PHI0, member=0)  # reported and cleared
