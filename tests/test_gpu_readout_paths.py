"""The readout where FP32 must leave the decision to FP64 and where its split
over CTAs has edges: equal and nearly equal largest pixels, pixels at the veto
threshold, no noise, one pixel to the largest grid, event counts around a
CTA's share, against the oracle."""
import numpy as np
import pytest

import oracle
import paper_2506_09712_gb300 as cts

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2506_09712_gb300 import build
    build.build()
    oracle.build()


@pytest.mark.parametrize("grid,n_ev", [(1, 3), (2, 29), (3, 28), (9, 57), (9, 1), (17, 30), (32, 9)])
@pytest.mark.parametrize("noise", [0.0, 0.13, 5.0])
def test_readout_matches_the_oracle(grid, n_ev, noise):
    rng = np.random.default_rng([grid, n_ev])
    counts = rng.poisson(0.3, (n_ev, grid, grid)).astype(np.int32)
    c = rng.integers(0, grid, (n_ev, 4))
    for k in range(n_ev):
        # two pixels that tie or differ by one count, of any size
        big = int(rng.choice([0, 3, 700, 5525, 2_000_000]))
        counts[k, c[k, 0], c[k, 1]] = big
        counts[k, c[k, 2], c[k, 3]] = big - int(rng.integers(0, 2)) * (big > 0)
    if n_ev > 2:
        counts[2] = 0                    # all pixels equal without noise
    seeds = rng.integers(1 << 62, size=n_ev).astype(np.uint64)
    ids = np.arange(n_ev, dtype=np.uint64) + (5 << 40)
    # a threshold of zero puts the ring's empty pixels on it
    for veto in (3.0, 0.0):
        for pixels in (False, True):
            kw = dict(noise_keV=noise, veto_factor=veto, window_keV=4.0)
            g = cts.sim_readout(counts, seeds, ids, 20.0, 300, want_pixels=pixels, **kw)
            o = oracle.readout(counts, seeds, ids, 20.0, 300, **kw)
            for k in ("cx", "cy", "vetoed", "accepted", "spectrum"):
                assert np.array_equal(g[k], o[k]), k
            # FP64 rounding of counts up to 7 MeV
            np.testing.assert_allclose(g["cluster"], o["cluster"], rtol=1e-13, atol=1e-12)
            np.testing.assert_allclose(g["e_cluster"], o["e_cluster"], rtol=1e-13, atol=1e-11)
            if pixels:
                np.testing.assert_allclose(g["e"], o["e"], rtol=1e-13, atol=1e-12)
