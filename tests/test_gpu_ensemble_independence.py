"""A member of an ensemble evolves as if the others were not there, to the last bit: how the columns are
cut into blocks depends on all members, the order of a member's sums on its own size only (and on the
pass kernel, which the ensemble's row alignment and largest member choose)."""
import numpy as np
import pytest

from tests.test_gpu_ensemble import member_params, run_ensemble

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def cl():
    from paper_2607_24978_gb300 import build_ext, cl as mod
    build_ext.build()
    mod.lib()
    return mod


# few and many members, in another order, beside larger and smaller ones; rows of vectors (staged
# passes) and of any alignment (direct ones); a size whose planes do not divide evenly
@pytest.mark.parametrize("size,others", [(64, ([64], [32] * 40, [48, 96])), (48, ([8], [64] * 200, [16, 32] * 9)),
                                         (20, ([20], [64] * 150)), (33, ([9], [17, 35] * 60)), (7, ([7], [31] * 300))])
@pytest.mark.parametrize("nf,prec", [(1, 0), (1, 1), (2, 1), (2, 2)])
def test_a_member_does_not_depend_on_the_others(cl, size, others, nf, prec):
    mine = member_params([size], nf, seed=size)[0]
    base = {n: member_params([n], nf, seed=n + 1)[0] for o in others for n in o}
    got = []
    for k, o in enumerate(others):
        rest = [base[n] for n in o]
        at = 0 if k % 2 == 0 else len(rest)
        out = run_ensemble(cl, rest[:at] + [mine] + rest[at:], nf, prec, 1, 0.02, 4)
        got.append((out[0][at], out[1][at], out[2][at]))
    for phi, pi, e in got[1:]:
        assert np.array_equal(phi, got[0][0]) and np.array_equal(pi, got[0][1])
        assert e == got[0][2]
