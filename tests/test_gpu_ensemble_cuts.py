"""The library's cuts of an ensemble into blocks of equal work against whole columns.

Cutting a column moves no field value; it reorders the FP64 sums of a and a', so the fields agree
to a few rounding errors a step (bound 1e-13 in FP64, as between other work-item shapes)."""
import pytest

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

