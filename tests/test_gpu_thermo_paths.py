"""rewl_thermo and rewl_thermo_jackknife where their kernel takes another path:
few and many CTAs, tables at the sizes where the threads of a CTA change and
where the weights no longer fit in shared memory, temperatures at which most
weights are zero or denormal, calls too large for the fixed scratch array, and
calls from several threads at once.  Tolerances: sums of n FP64 terms with a
weight good to about one unit in the last place, n * 2^-52 and a factor for the
cancellation in F and S; 1e-10 covers all of it, as in test_gpu_thermo.py."""
import threading

import numpy as np
import pytest

from oracle.thermo import jackknife, thermodynamics
from paper_1305_5615_gb300 import rewl

pytestmark = pytest.mark.gpu


def table(n, seed):
    rng = np.random.default_rng(seed)
    p = np.clip(np.linspace(0.0, 1.0, n), 1e-9, 1 - 1e-9)
    g = -n * (p * np.log(p) + (1 - p) * np.log(1 - p)) + 1.0 + 0.01 * rng.standard_normal(n)
    if n > 4:
        g[1] = g[-2] = -np.inf
    return g


@pytest.mark.parametrize("n", [1, 31, 65, 2048, 2049, 4096, 4097, 8193])
@pytest.mark.parametrize("n_T", [1, 305])
def test_sizes(n, n_T):
    g, T = table(n, n), np.concatenate([[0.02], np.linspace(0.3, 50.0, n_T - 1)]) if n_T > 1 else np.array([2.5])
    got, ref = rewl.rewl_thermo(g, -2 * (n - 1), 4, T), thermodynamics(g, -2 * (n - 1), 4, T)
    assert np.allclose(got, ref, rtol=1e-10, atol=1e-9)


def test_a_call_larger_than_the_scratch_array():
    runs = np.stack([table(8193, s) for s in range(10)])
    T = np.linspace(1.0, 4.0, 70)
    est, err = rewl.rewl_thermo_jackknife(runs, -16384, 4, T)
    e_ref, r_ref = jackknife(runs, -16384, 4, T)
    assert np.allclose(est, e_ref, rtol=1e-10, atol=1e-9)
    assert np.allclose(err, r_ref, rtol=1e-6, atol=1e-9)


def test_calls_from_several_threads():
    T = np.linspace(0.5, 5.0, 40)
    tables = [table(300 + 7 * i, i) for i in range(8)]
    ref = [rewl.rewl_thermo(g, -600, 4, T) for g in tables]
    bad = []

    def work(i):
        for _ in range(20):
            if not np.array_equal(rewl.rewl_thermo(tables[i], -600, 4, T), ref[i]):
                bad.append(i)

    ts = [threading.Thread(target=work, args=(i,)) for i in range(8)]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    assert not bad
