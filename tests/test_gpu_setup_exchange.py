"""The set-up walks (32 moves decided together) and the exchange (configurations
swapped by warps) against the oracle, bit for bit, at sizes where they can go
wrong: neighbours that coincide, packed rows with a remainder, configurations of
one word and of many, walks that run out of their budget and start again, odd
window counts, a single window (no pair, the clocks move on by themselves), and
walkers per window that do not fill the warps."""
import pytest

from oracle import OracleREWL
from paper_1305_5615_gb300 import rewl
from parity_util import compare_states, make_pair, run_both

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("model,L,q,h,m,entry", [("ising", 2, 2, 1, 1, 1000), ("ising", 31, 2, 5, 3, 1000),
                                                 ("ising", 33, 2, 6, 2, 20), ("ising", 64, 2, 9, 1, 3),
                                                 ("potts", 3, 16, 1, 33, 1000), ("potts", 9, 2, 2, 5, 50),
                                                 ("potts", 25, 11, 7, 3, 10), ("ea", 10, 2, 3, 4, 1000),
                                                 ("ea", 34, 2, 4, 2, 300), ("ea3d", 6, 2, 3, 3, 1000)])
def test_setup(model, L, q, h, m, entry):
    O, D = make_pair(model, L, h, 0.75, m, 0.8, 1e-6, 40 + L, q=q, entry_max_sweeps=entry, discovery_sweeps=7)
    assert compare_states(O, D, "set-up") == 0


def test_a_walk_that_cannot_enter_fails_on_both_sides():
    args = ("ising", 32, 16, 0.75, 1, 0.8, 1e-6, 1)     # the top window is far from the ground state: one sweep is too few
    with pytest.raises(RuntimeError):
        OracleREWL(*args, entry_max_sweeps=1)
    with pytest.raises(rewl.RewlError) as e:
        rewl.REWL(*args, entry_max_sweeps=1)
    assert e.value.status == 5


@pytest.mark.parametrize("model,L,q,h,m", [("ising", 6, 2, 2, 130), ("ising", 40, 2, 5, 3), ("potts", 17, 5, 3, 37),
                                           ("ea", 12, 2, 3, 1), ("ea3d", 8, 2, 4, 2), ("ising", 8, 2, 1, 4)])
@pytest.mark.parametrize("mode", [rewl.MODE_PLAIN, rewl.MODE_GRAPH])
def test_exchange_every_sweep(model, L, q, h, m, mode):
    """Sixteen exchange rounds, one a sweep, with a flatness check every four."""
    O, D = make_pair(model, L, h, 0.75, m, 0.8, 1e-6, 7, q=q, spe=1, spf=4, mode=mode)
    run_both(O, D, 16, 1)
    assert compare_states(O, D, "16 rounds") == 0
    if h > 1:
        assert int(D.state()["x_accepted"].sum()) > 0
