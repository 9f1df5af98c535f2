"""Binned spectra against numpy's FFT and a histogram: sizes with and without Nyquist rows, rows
shorter and longer than a warp, bins wider and narrower than a mode (the last case has more bins
than the block's histogram holds), and a handle whose kept scratch grows and shrinks with the
member.  FP64 transforms of these sizes agree to a few 1e-15 of the largest amplitude; a bin sums
powers of one shell, so 1e-12 of the bin with a floor of 1e-12 of the largest bin."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def cl():
    from paper_2607_24978_gb300 import build_ext, cl as mod
    build_ext.build()
    mod.lib()
    return mod


def reference(f, L, dn, type_):
    N = f.shape[0]
    P = np.abs(np.fft.fftn(f)) ** 2
    i = np.arange(N)
    s = np.where(i <= N // 2, i, i - N).astype(float)
    nm = np.sqrt(s[:, None, None] ** 2 + s[None, :, None] ** 2 + s[None, None, :] ** 2)
    l = np.floor(nm / dn + 0.5).astype(np.int64).ravel()
    nb = int(np.floor(np.sqrt(3.0) * (N // 2) / dn + 0.5)) + 1
    S = np.bincount(l, P.ravel(), nb)[:nb]
    C = np.bincount(l, minlength=nb)[:nb].astype(float)
    n = np.arange(nb) * dn
    with np.errstate(divide="ignore", invalid="ignore"):
        d = n * S / (float(N) ** 6 * dn) if type_ == 1 else 4 * np.pi * n ** 3 * (S / C) / float(N) ** 6
    return 2 * np.pi / L * n, np.where((n > 0) & (C > 0), d, 0.0), C


def check(got, want):
    (k, d, c), (k2, d2, c2) = got, want
    assert np.array_equal(c, c2)
    assert np.allclose(k, k2, rtol=1e-14)
    assert np.allclose(d, d2, rtol=1e-12, atol=1e-12 * d2.max())


@pytest.mark.parametrize("N", [2, 3, 4, 5, 16, 33, 64, 65, 100])
@pytest.mark.parametrize("dn,type_", [(1.0, 1), (1.0, 2), (2.5, 1), (0.7, 2), (0.01, 1)])
def test_against_numpy(cl, N, dn, type_):
    f = 1.0 + np.random.default_rng(N).standard_normal((N, N, N))
    with cl.Lattice(N, 3.0, 1, cl.CL_PREC_FP64, cl.CL_INT_VV2) as g:
        g.cl_set_potential(cl.CL_POT_LPHI4, [1.0])
        g.cl_set_state(cl.CL_FIELD_PHI0, f)
        want = reference(f, 3.0, dn, type_)
        check(g.cl_spectrum(cl.CL_FIELD_PHI0, dn, type_), want)
        check(g.cl_spectrum(cl.CL_FIELD_PHI0, dn, type_), want)  # from the kept plan and scratch


def test_members_of_many_sizes_share_the_scratch(cl):
    sizes = [8, 24, 10, 6, 12, 14, 16, 18, 20, 22, 9, 24, 8]  # more sizes than plans are kept
    g = np.random.default_rng(3)
    with cl.Lattice(8, 3.0, 1, cl.CL_PREC_FP64, cl.CL_INT_VV2, member_N=sizes) as lat:
        lat.cl_set_potential(cl.CL_POT_LPHI4, [1.0])
        fields = [g.standard_normal((n, n, n)) for n in sizes]
        for m, f in enumerate(fields):
            lat.cl_set_state(cl.CL_FIELD_PHI0, f, member=m)
        for m in list(range(len(sizes))) + [0, 5]:
            check(lat.cl_spectrum(cl.CL_FIELD_PHI0, member=m), reference(fields[m], 3.0, 1.0, 1))
