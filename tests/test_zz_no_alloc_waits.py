"""rewl_sweep_noalloc with few walkers: its ring form waits between the warps of
a walker, each wait bounded.  A wait that runs out is told in the walker's
status; the bound grows with the trials of the call, so a long call does not run
it out.  (Its constant part is given through rewl_sweep_noalloc_waits, which the
library has for this test; the waits end by themselves or give up.)  Above that
walker count the call runs the form without waits."""
import ctypes

import numpy as np
import pytest

from paper_1305_5615_gb300 import rewl
from test_zz_no_alloc import _desc, _device_state

pytestmark = pytest.mark.gpu

L, M, SWEEPS = 20, 6, 1000       # 400 000 trials a walker: some 10^7 cycles
GROWTH = SWEEPS * L * L << 10    # of the bound, for that many trials


def run(wait_cycles):
    """Statuses and state of six walkers of one window after 1000 sweeps with the given bound."""
    import torch

    D = rewl.REWL("ising", L, 1, 0.75, M, 0.8, 1e-6, 9)
    dev = _device_state(torch, D.state())
    lat, E, lng, H, win, lnf = dev
    status = torch.full((M,), -1, dtype=torch.int32, device="cuda")
    desc = _desc(D.info, L, 1, M, 9, SWEEPS, 0, status.data_ptr())
    f = rewl.load().rewl_sweep_noalloc_waits
    f.argtypes = [ctypes.c_void_p] * 9 + [ctypes.c_longlong]
    assert f(ctypes.byref(desc), lat.data_ptr(), E.data_ptr(), lng.data_ptr(), H.data_ptr(), None, win.data_ptr(),
             lnf.data_ptr(), None, wait_cycles) == 0
    torch.cuda.synchronize()
    return status.cpu().numpy(), [x.cpu().numpy() for x in (lat, E, lng, H)]


def test_a_wait_that_runs_out_is_told_in_the_status():
    status, (lat, E, _, H) = run((1 << 20) - GROWTH)    # 2^20 cycles in all: far less than the call takes
    assert (status == 4).all()               # REWL_ETIMEOUT
    visits = H.reshape(M, -1).sum(1)
    assert (visits < SWEEPS * L * L).all() and (visits % 32 == 0).all()
    s = 1 - 2 * rewl.unpack_lattice(lat.view(np.uint32).reshape(M, -1), L, rewl.ISING).reshape(M, L, L).astype(int)
    assert np.array_equal(E, -(s * (np.roll(s, 1, 1) + np.roll(s, 1, 2))).sum((1, 2)))   # an earlier trial's state


def test_the_length_of_the_call_does_not_run_a_wait_out():
    import torch

    status, got = run(1 << 20)
    assert (status == 0).all()
    D = rewl.REWL("ising", L, 1, 0.75, M, 0.8, 1e-6, 9)
    lat, E, lng, H, win, lnf = _device_state(torch, D.state())
    rewl.rewl_sweep_noalloc(_desc(D.info, L, 1, M, 9, SWEEPS, 8), lat.data_ptr(), E.data_ptr(), lng.data_ptr(),
                            H.data_ptr(), None, win.data_ptr(), lnf.data_ptr(), None)   # 8 lanes: no waits
    torch.cuda.synchronize()
    for a, b in zip(got, (lat, E, lng, H)):
        assert np.array_equal(a.view(np.uint8), b.cpu().numpy().view(np.uint8))


@pytest.mark.parametrize("model,q", [("ising", 2), ("potts", 5), ("ea", 2)])
def test_more_walkers_than_the_ring_form_runs_in_one_wave(model, q):
    import torch

    from oracle import OracleREWL
    from test_zz_no_alloc import _coupling_bits, _to_dev

    m = 2 * torch.cuda.get_device_properties(0).multi_processor_count    # 8 an SM; the ring form holds at most 7
    D = rewl.REWL(model, 8, 4, 0.75, m, 0.8, 1e-6, 13, q=q)
    bits = None
    if model == "ea":
        bits = _to_dev(torch, _coupling_bits(OracleREWL(model, 8, 4, 0.75, 1, 0.8, 1e-6, 13).couplings(), 8), np.int32)
    got = []
    for lanes in (0, 8):
        lat, E, lng, H, win, lnf = _device_state(torch, D.state())
        rewl.rewl_sweep_noalloc(_desc(D.info, 8, 4, m, 13, 50, lanes), lat.data_ptr(), E.data_ptr(), lng.data_ptr(),
                                H.data_ptr(), bits.data_ptr() if bits is not None else None, win.data_ptr(),
                                lnf.data_ptr(), None)
        torch.cuda.synchronize()
        got.append([x.cpu().numpy().view(np.uint8) for x in (lat, E, lng, H)])
    assert all(np.array_equal(a, b) for a, b in zip(*got))


def test_a_window_that_only_fits_the_sequential_chain():
    """28 915 bins: 232 408 bytes for the chain with a whole warp, 232 544 with the other forms' tables; a CTA has
    232 448.  Against 8 lanes."""
    import torch

    D = rewl.REWL("ising", 16, 1, 0.75, 3, 0.8, 1e-6, 21)
    st, bins = D.state(), 28915
    got = []
    for lanes in (0, 8):
        lat, E, _, _, win, lnf = _device_state(torch, st)
        lng = torch.zeros(3 * bins, dtype=torch.float64, device="cuda")
        H = torch.zeros(3 * bins, dtype=torch.int32, device="cuda")
        desc = _desc(dict(D.info, window_bins=bins), 16, 1, 3, 21, 20, lanes)
        rewl.rewl_sweep_noalloc(desc, lat.data_ptr(), E.data_ptr(), lng.data_ptr(), H.data_ptr(), None,
                                win.data_ptr(), lnf.data_ptr(), None)
        torch.cuda.synchronize()
        assert int(H.sum()) == 3 * 20 * 256
        got.append([x.cpu().numpy().view(np.uint8) for x in (lat, E, lng, H)])
    assert all(np.array_equal(a, b) for a, b in zip(*got))
