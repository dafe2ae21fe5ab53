"""Fast generation where its two paths meet: events around a warp's and a
CTA's share of carriers (the queue of undecided carriers drains partly
filled), shapes that reject often, pixels much smaller and much larger than
the cloud (every carrier, or none, near an edge), against the FP64 sampler."""
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
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


@pytest.mark.parametrize("beta", [0.5, 1.0, 2.4, 6.0])
@pytest.mark.parametrize("pitch,grid", [(25.0, 9), (0.8, 32), (2000.0, 1)])
def test_counts_match_the_oracle_sampler(beta, pitch, grid):
    sizes = (0, 1, 31, 32, 33, 63, 64, 255, 256, 257, 511, 1000, 5525)
    evs = [dict(seed=77, event_id=(3 << 33) + k, n_pairs=n, x_um=1.5 - 0.4 * k, y_um=0.3 * k - 2.0,
                alpha=6.0, beta=beta) for k, n in enumerate(sizes)]
    gp, go = cts.sim_generate(evs, pitch, grid)
    op, oo = oracle.generate(evs, pitch, grid)
    n = np.array(sizes)
    assert np.array_equal(gp.reshape(len(evs), -1).sum(1) + go, n)
    # FP32 draws move a carrier across an edge now and then: at most two per
    # pixel (the bound of the generation tests), few events at all
    d = np.abs(gp.astype(np.int64) - op).reshape(len(evs), -1)
    assert d.max() <= 2 and np.abs(go - oo).max() <= 2
    assert d.sum() <= 2e-4 * n.sum() * (32 if pitch < 1.0 else 1)
