"""The symmetric kernel's finer units (few events with enough pair work for
it) against the FP64 oracle: one step of single events of each size class,
both species, partly filled blocks and tiles."""
import numpy as np
import pytest

import oracle
import paper_2506_09712_gb300 as cts
import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_h,n_e", [(5525, 0), (4001, 3999), (20_500, 0), (11_003, 10_007),
                                     (41_001, 0)])
def test_one_step_matches_the_oracle(n_h, n_e):
    from paper_2506_09712_gb300 import build
    build.build()
    oracle.build()
    p = W.preset("track_200keV_320um")
    params = oracle.make_params(p["sensor"], W.field_switches(), p["mobility"])
    n = n_h + n_e
    xyz = W.random_cloud(n, 4.0, center=(1.0, -2.0, 160.0), seed=n)
    xyz[n_h:, 2] += 5.0
    sign = np.where(np.arange(n) < n_h, 1, -1).astype(np.int8)
    o_pos, o_st = oracle.step(params, 7, 3, 0, xyz, sign, np.zeros(n, dtype=np.int8))
    d = np.linalg.norm(o_pos - xyz, axis=1)
    for variant in (1, 13):
        with cts.Simulator(p["sensor"], p["mobility"], max_slots=4, variant=variant) as sim:
            g_pos, g_st = cts.sim_debug_step(sim.h, 7, 3, xyz, sign)
        assert np.array_equal(g_st, o_st)
        rel = np.linalg.norm(g_pos - o_pos, axis=1) / d
        # the bounds of the one-step parity tests (FP32 arithmetic of the step)
        assert np.median(rel) < 4e-7
        assert rel.max() < 2e-4
