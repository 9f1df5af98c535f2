"""Tiling options and the autotuner beside the kernels that the library chooses by itself: rows of any
alignment, and resident launches of small lattices."""
import numpy as np
import pytest

from tests import inputs

pytestmark = pytest.mark.gpu
OPTIONS = ("CL_OPT_STAGES", "CL_OPT_TILE_BY", "CL_OPT_TILE_DZ", "CL_OPT_PASS_VARIANT")


@pytest.fixture(scope="module")
def cl():
    from paper_2607_24978_gb300 import build_ext, cl as mod
    build_ext.build()
    mod.lib()
    return mod


def lattice(cl, N, prec=1):
    phi, pi = inputs.scalar_state(N, 1, seed=N, fbar=(1.0,), amp=0.05, pamp=0.05)
    dtype = np.float64 if prec == 0 else np.float32
    g = cl.Lattice(N, 0.4 * N, 1, prec, cl.CL_INT_VV2, expansion=True, alpha=0.3, kappa=0.2, dt=0.01)
    g.cl_set_potential(cl.CL_POT_LPHI4, [1.0])
    g.cl_set_state(cl.CL_FIELD_PHI0, phi[0].astype(dtype))
    g.cl_set_state(cl.CL_FIELD_PI0, pi[0].astype(dtype))
    g.cl_set_scalars(1.0)
    return g


@pytest.mark.parametrize("N", [33, 34, 161])
@pytest.mark.parametrize("option", OPTIONS)
def test_setting_what_is_reported_changes_no_tiling(cl, N, option):
    with lattice(cl, N) as g:
        before = [g.cl_get_option(getattr(cl, o)) for o in OPTIONS]
        g.cl_set_option(getattr(cl, option), g.cl_get_option(getattr(cl, option)))
        assert [g.cl_get_option(getattr(cl, o)) for o in OPTIONS] == before
        assert before[0] in (3, 4)


def numbers(cl, g, steps=40):
    """FP64 sums and a(t) of a run: the order of the sums, hence the kernel, is in their last bits."""
    out = []
    for _ in range(steps):
        g.cl_step(1)
        e = g.cl_energies()
        out += [e[k] for k in ("a", "adot", "K0", "G0", "V")]
    return out


def test_the_resident_launches_are_the_tuners_choice_and_stay_so(cl, tmp_path):
    """At 16^3 a resident pass takes a quarter of a launch: the tuner keeps it, reports its time, and
    an option set back to the library's choice afterwards does not end it."""
    with lattice(cl, 16, 0) as g:
        plain = numbers(cl, g)
    with lattice(cl, 16, 0) as g:
        g.cl_set_option(cl.CL_OPT_TILE_BY, 3)
        tiled = numbers(cl, g)
    assert plain != tiled
    cache = str(tmp_path / "tune.jsonl")
    for again in (False, True):  # trials, then the choice read back
        with lattice(cl, 16, 0) as g:
            state = g.cl_get_state(cl.CL_FIELD_PHI0), g.cl_get_state(cl.CL_FIELD_PI0), g.cl_get_scalars()
            us = g.cl_autotune(cache)[3]
            assert 0.0 < us < 9.0  # a launch per pass takes 12 us and more
            after = g.cl_get_state(cl.CL_FIELD_PHI0), g.cl_get_state(cl.CL_FIELD_PI0), g.cl_get_scalars()
            assert np.array_equal(state[0], after[0]) and np.array_equal(state[1], after[1]) and state[2] == after[2]
            g.cl_set_option(cl.CL_OPT_TILE_DZ, 0)
            assert numbers(cl, g) == plain
    assert '"resident": 1' in open(cache).read()


def test_a_tuned_choice_of_launches_is_kept(cl, tmp_path):
    """A cached choice that found a launch per pass faster runs one; a line without that word, as files
    written before it have, leaves the library's choice."""
    key = '{"key": "single N=16 nf=1 prec=0", "stages": -1, "by": 3, "dz": 0, "variant": 0, "us": 1.000%s}\n'
    runs = []
    for word in (', "resident": 0', ""):
        cache = tmp_path / "tune.jsonl"
        cache.write_text(key % word)
        with lattice(cl, 16, 0) as g:
            g.cl_autotune(str(cache))
            runs.append(numbers(cl, g))
    with lattice(cl, 16, 0) as g:
        assert runs[1] == numbers(cl, g)
    with lattice(cl, 16, 0) as g:
        g.cl_set_option(cl.CL_OPT_TILE_BY, 3)
        assert runs[0] == numbers(cl, g)


def test_the_tuner_puts_an_open_leapfrog_back(cl):
    with lattice(cl, 20) as g, lattice(cl, 20) as h:
        for x in (g, h):
            x.cl_step(5)
        g.cl_autotune()
        for x in (g, h):
            x.cl_set_option(cl.CL_OPT_TILE_BY, 4)
            x.cl_set_option(cl.CL_OPT_TILE_DZ, 5)
            x.cl_set_option(cl.CL_OPT_STAGES, -1)
            x.cl_set_option(cl.CL_OPT_PASS_VARIANT, 0)
            x.cl_step(3)
        assert g.cl_energies() == h.cl_energies()
        for f in (cl.CL_FIELD_PHI0, cl.CL_FIELD_PI0):
            assert np.array_equal(g.cl_get_state(f), h.cl_get_state(f))
