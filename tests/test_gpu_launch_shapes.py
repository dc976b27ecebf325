"""Which form a solve runs in and with which launch shape, where an option or a
forced shape meets the automatic choice; the states are the same bits in every
form."""
import ctypes

import numpy as np
import pytest

from paper_1305_5615_gb300 import rewl
from parity_util import compare_states, make_pair, run_both

pytestmark = pytest.mark.gpu


def n_sm():
    import torch

    return torch.cuda.get_device_properties(0).multi_processor_count


def same_states(A, B):
    a, b = A.state(), B.state()
    for k in ("lattice", "E", "H", "lnf", "iteration", "wl_accept", "x_accepted"):
        assert np.array_equal(a[k], b[k]), k
    assert np.array_equal(a["lng"].view(np.uint64), b["lng"].view(np.uint64))


@pytest.mark.parametrize("per_sm,variant,lanes,expect", [
    (7, -1, 0, (0, 32, 0)),    # automatic: the form that decides 32 trials together, which takes no prepared draws
    (9, -1, 0, (0, 32, 0)),
    (9, -1, 8, (0, 8, 1)),     # lanes that only the sequential chain has
    (9, 0, 0, (0, 32, 1)),     # the chain asked for: prepared draws, a whole warp up to 12 walkers an SM
    (13, 0, 0, (0, 8, 1)),
    (33, 0, 0, (0, 32, 0)),    # too many walkers for prepared draws
])
def test_prepared_draws_leave_the_faster_forms_alone(per_sm, variant, lanes, expect):
    m = -(-per_sm * n_sm() // 4)
    kw = dict(lanes_per_walker=lanes, sweeps_per_exchange=20, sweeps_per_flat_check=100)
    A = rewl.REWL("ising", 8, 4, 0.75, m, 0.8, 1e-8, 5, sweep_variant=variant, prefetch_draws=1, **kw)
    got = A.info["sweep_variant"], A.info["lanes_per_walker"], A.info["prefetch_draws"]
    assert got == expect
    B = rewl.REWL("ising", 8, 4, 0.75, m, 0.8, 1e-8, 5, sweep_variant=1, **kw)
    for D in (A, B):
        D.step(200)
    same_states(A, B)


def test_sweeps_with_prepared_draws_take_as_long_queued_as_one_at_a_time():
    """Ten blocks queued back to back against blocks waited for one by one: the kernel that prepares draws does not
    take the sweeps' places on the chip (it once doubled their time; the bound leaves room for the walk itself)."""
    D = rewl.REWL("ising", 32, 16, 0.75, 4, 0.8, 1e-8, 5, sweep_variant=0, prefetch_draws=1, profile=True)
    assert D.info["prefetch_draws"] == 1
    D.step(100)
    t0 = D.info["sweep_ms"]
    for _ in range(9):
        D.step(100)
    t1 = D.info["sweep_ms"]
    D.step(1000)
    one, queued = (t1 - t0) / 9, (D.info["sweep_ms"] - t1) / 10
    assert queued < 1.3 * one, (one, queued)


def test_walkers_per_block_is_charged_at_the_lanes_it_was_always_charged_at():
    """More than 8 walkers an SM with walkers per block asked for and lanes left open: accepted by the shared memory of
    8 lanes a walker (8 x (8 B x (bins + 16) + 4 B x 128 words + 28 B x 8 trials) at L = 64), refused beyond, whatever
    the form that runs takes; the walkers per block that are reported are those that run."""
    m = -(-9 * n_sm() // 2)

    def create(bins, wpb):
        return rewl.REWL("ising", 64, 2, 0.75, m, 0.8, 1e-8, 5, walkers_per_block=wpb,
                         window_starts=[0, 4097 - bins], window_widths=[bins, bins])

    most = (227 * 1024 // 8 - 28 * 8 - 4 * 128) // 8 - 16
    D = create(most, 8)
    assert (D.info["lanes_per_walker"], D.info["walkers_per_block"], D.info["sweep_variant"]) == (32, 2, 0)
    D.close()
    for bins, wpb in ((most + 1, 8), (2100, 16)):     # 16 walkers of 1764 bins are the most that fit
        with pytest.raises(rewl.RewlError) as e:
            create(bins, wpb)
        assert e.value.status == 1


@pytest.mark.parametrize("prefetch", [0, 1])
def test_windows_that_only_fit_the_sequential_chain(prefetch):
    """24 500 bins of Potts on 256 x 256: 229 792 bytes for the chain with a whole warp, 232 864 with the tables of the
    forms that decide 32 trials together, and a CTA has 232 448; its draws may be prepared ahead."""
    O, D = make_pair("potts", 256, 6, 0.130016, 1, 0.8, 1e-6, 2, q=10, spe=1, spf=2, prefetch_draws=prefetch)
    i = D.info
    assert (i["window_bins"], i["sweep_variant"], i["lanes_per_walker"], i["prefetch_draws"]) == (24500, 0, 32, prefetch)
    run_both(O, D, 3, 1)
    assert compare_states(O, D, "24500 bins") == 0


def test_autotune_returns_what_it_timed():
    """The candidates are timed without prepared draws, so the best is returned without them: 9 walkers an SM take the
    chain with a whole warp, which with them is the sequential form."""
    m = -(-9 * n_sm() // 4)
    p, best = rewl.rewl_params_default(), rewl.rewl_params()
    p.sweeps_per_exchange, p.sweeps_per_flat_check, p.prefetch_draws = 20, 100, 1
    res, n = (rewl.rewl_tune_result * 8)(), ctypes.c_int32()
    args = (rewl.rewl_model(0, 2), rewl.rewl_lattice(2, 8, 8, 1))
    assert rewl.load().rewl_autotune(ctypes.byref(args[0]), ctypes.byref(args[1]), None, 4, 0.75, m, 0.8, 1e-8,
                                     ctypes.c_uint64(5), ctypes.byref(p), 40, res, 8, ctypes.byref(n),
                                     ctypes.byref(best)) == 0
    h = rewl.rewl_create(*args, None, 4, 0.75, m, 0.8, 1e-8, 5, best)
    i = rewl.rewl_get_info(h)
    rewl.rewl_destroy(h)
    assert i["prefetch_draws"] == 0
    assert (i["sweep_variant"], i["lanes_per_walker"]) == (best.sweep_variant, best.lanes_per_walker)
