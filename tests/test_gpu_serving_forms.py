"""Served form: a bounded wait of the batched ring sweeps that runs out fails its
request, and every sweep form of a round gives the bits of the solve alone."""
import numpy as np
import pytest

from paper_1305_5615_gb300 import rewl

pytestmark = pytest.mark.gpu


def test_a_wait_that_runs_out_fails_the_request():
    """With a bound of a few cycles the first wait that finds its batch not ready gives up and the walkers of the
    request stop part way: it fails with REWL_ETIMEOUT and holds nothing, and the next server serves it."""
    for wait_cycles, state, error in ((4, rewl.REQ_FAILED, 4), (0, rewl.REQ_DONE, 0)):
        S = rewl.RewlServer(device_bytes=1 << 30, max_running=4, wait_cycles=wait_cycles)
        rid = S.submit("ising", 8, 4, 0.75, 2, 0.8, 1e-2, 11)
        for _ in range(500):
            st = S.run(20)
            if st["running"] == 0:
                break
        info = S.poll(rid)
        assert (info["state"], info["error"]) == (state, error)
        assert st["device_bytes_in_use"] == 0 and st["failed"] == (error != 0)
        S.close()


def finish(S, ids):
    for _ in range(2000):
        st = S.run(20)
        if st["running"] + st["queued"] == 0:
            break
    assert st["finished"] == len(ids) and st["failed"] == 0
    return [S.result(i, 1 << 17)[0].view(np.uint64) for i in ids]


@pytest.mark.parametrize("model,L,q", [("potts", 5, 7), ("ea", 6, 2), ("ea3d", 4, 2)])
def test_full_server_makes_its_own_draws(model, L, q):
    """Forty requests of 32 walkers, more than 5 an SM: no producer warps."""
    reqs = [(model, L, 4, 0.75, 8, 0.8, 0.1, 500 + i) for i in range(40)]
    S = rewl.RewlServer(device_bytes=4 << 30, max_running=64)
    got = finish(S, [S.submit(*r, q=q) for r in reqs])
    for i in (0, 17, 39):
        D = rewl.REWL(*reqs[i], q=q)
        assert D.step(0)
        assert np.array_equal(got[i], D.lng()[0].view(np.uint64)), i


def test_windows_that_only_fit_the_sequential_chain():
    """27 600 bins of Potts on 128 x 128: 230 016 bytes for the chain, 232 064 with the other forms' tables, and a
    round's kernels have 231 424.  Flatness 1e-6 passes at once, so that the solve ends after a few checks."""
    kw = dict(sweeps_per_exchange=2, sweeps_per_flat_check=2)
    req = ("potts", 128, 2, 0.8127, 2, 1e-6, 0.2, 3)
    S = rewl.RewlServer(device_bytes=1 << 30, max_running=2, **kw)
    got, = finish(S, [S.submit(*req, q=4)])
    D = rewl.REWL(*req, q=4, **kw)
    assert D.info["window_bins"] == 27600
    assert D.step(0)
    assert np.array_equal(got, D.lng()[0].view(np.uint64))
