"""Served form: a bounded wait of the batched ring sweeps that runs out fails its
request, and every sweep form of a round gives the bits of the solve alone."""
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
