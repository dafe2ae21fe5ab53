"""Stateless entry points that keep device memory between calls: calls of
growing and shrinking size, from several threads at once, around handles that
come and go, give the results of a first call."""
import threading

import numpy as np
import pytest

import paper_2506_09712_gb300 as cts
import workloads as W

pytestmark = pytest.mark.gpu


def _call(n, seed):
    rng = np.random.default_rng(seed)
    rec = cts.gen_events(seed, np.arange(n), rng.integers(1, 900, n), rng.uniform(-9, 9, n),
                         rng.uniform(-9, 9, n), 5.0, 2.4)
    pix, out = cts.sim_generate(rec, 25.0, 9)
    r = cts.sim_readout(pix, np.full(n, seed), np.arange(n), 2.0, n_bins=50, want_pixels=True)
    return [pix, out] + [r[k] for k in ("e", "cluster", "accepted", "cx", "cy", "spectrum")]


def _same(a, b):
    return all(np.array_equal(x, y, equal_nan=x.dtype.kind == "f") for x, y in zip(a, b))


def test_calls_of_any_size_and_thread_agree_with_a_first_call():
    sizes = (1, 700, 3, 4000, 28, 1, 2500)
    first = {n: _call(n, 5) for n in set(sizes)}
    for n in sizes:
        assert _same(_call(n, 5), first[n])
    p = W.preset("plain_3keV_100um")
    bad = []

    def work(k):
        for n in sizes[k % 3:]:
            if k == 1:  # a handle made and destroyed beside the calls
                with cts.Simulator(p["sensor"], p["mobility"], max_slots=2):
                    pass
            if not _same(_call(n, 5), first[n]):
                bad.append((k, n))

    threads = [threading.Thread(target=work, args=(k,)) for k in range(6)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not bad
