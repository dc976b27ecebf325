"""The sweep forms that decide 32 trials together (the ring form and, with 32
lanes, the chain form) against the oracle, bit for bit, where they can go wrong:
lattices whose neighbours coincide (L = 2), ragged last groups, both sides of the
site count from which trials that touch one another come as pairs (400), both
sides of the ln f from which visits are counted in every group (2^-9), very large
and very small ln f, windows a few bins wide, and each model."""
import numpy as np
import pytest

from paper_1305_5615_gb300 import rewl
from parity_util import compare_states, make_pair, run_both

pytestmark = pytest.mark.gpu

FORMS = {"ring": dict(sweep_variant=2), "own draws": dict(sweep_variant=0, lanes_per_walker=32)}


def check(form, model, L, q, h, m, lnf0, blocks=4, spe=25, seed=None, **kw):
    """Four blocks of 25 sweeps; the last blocks follow a flatness check and the exchanges."""
    forms = dict(FORMS[form])
    G = forms.pop("lanes_per_walker", 0)
    O, D = make_pair(model, L, h, 0.75, m, 0.8, 1e-11, 1000 + L if seed is None else seed, q=q, spe=spe, spf=2 * spe,
                     lnf0=lnf0, G=G, **forms, **kw)
    where = "%s %s L=%d q=%d lnf0=%g" % (form, model, L, q, lnf0)
    assert compare_states(O, D, where + " entry") == 0
    run_both(O, D, blocks, spe)
    assert compare_states(O, D, where) == 0
    return D


@pytest.mark.parametrize("form", list(FORMS))
@pytest.mark.parametrize("model,L,q,h", [("ising", 2, 2, 1), ("ising", 3, 2, 1), ("potts", 2, 16, 1), ("potts", 5, 2, 2),
                                         ("ea", 2, 2, 1), ("ea3d", 2, 2, 1), ("ea3d", 4, 2, 2), ("ising", 19, 2, 4),
                                         ("ising", 20, 2, 4), ("potts", 19, 7, 3), ("potts", 21, 3, 3), ("ea", 20, 2, 3),
                                         ("ea3d", 8, 2, 3), ("ising", 65, 2, 8)])
def test_small_odd_and_both_sides_of_the_pairs(form, model, L, q, h):
    check(form, model, L, q, h, 2, 1.0, seed=4 if L == 2 else None)   # seed 4: couplings with a negative energy


@pytest.mark.parametrize("form", list(FORMS))
@pytest.mark.parametrize("lnf0", [64.0, 2.0 ** -8, 2.0 ** -9, 2.0 ** -20, 2.0 ** -36])
@pytest.mark.parametrize("model,L,q", [("ising", 12, 2), ("ising", 24, 2), ("potts", 22, 10)])
def test_every_ln_f(form, lnf0, model, L, q):
    check(form, model, L, q, 3, 2, lnf0)


@pytest.mark.parametrize("form", list(FORMS))
def test_narrow_windows(form):
    starts = np.arange(0, 101, 2, dtype=np.int32)
    widths = np.full(starts.size, 5, np.int32)      # five bins a window, three shared
    widths[-1] = 145 - starts[-1]
    check(form, "ising", 12, 2, starts.size, 1, 1.0, window_starts=starts, window_widths=widths)


def test_many_walkers_run_the_form_with_own_draws():
    """More walkers than the ring form runs in one wave: 32 lanes, chain variant, same bits as the ring form."""
    A = rewl.REWL("ising", 10, 8, 0.75, 160, 0.8, 1e-8, 3)
    B = rewl.REWL("ising", 10, 8, 0.75, 160, 0.8, 1e-8, 3, sweep_variant=2)
    assert (A.info["sweep_variant"], A.info["lanes_per_walker"]) == (0, 32)
    for D in (A, B):
        D.step(1000)
    a, b = A.state(), B.state()
    for k in ("lattice", "E", "H", "lnf", "wl_accept", "exact_tests", "x_accepted"):
        assert np.array_equal(a[k], b[k]), k
    assert np.array_equal(a["lng"].view(np.uint64), b["lng"].view(np.uint64))
