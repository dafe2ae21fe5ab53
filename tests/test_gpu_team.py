"""The team kernel (the default while few events run) against the FP64 oracle
where its partition changes: one carrier, partly filled rows of four, source
segments of 64 around their ends, fewer rows than warps, both species, and
events that shrink to nothing while others run on."""
import numpy as np
import pytest

import oracle
import paper_2506_09712_gb300 as cts
import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2506_09712_gb300 import build
    build.build()
    oracle.build()
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


@pytest.mark.parametrize("n_h,n_e", [(1, 0), (4, 0), (5, 0), (63, 0), (64, 1), (65, 64), (130, 127),
                                     (515, 0), (829, 0), (1, 700), (2001, 1500), (8191, 0)])
def test_one_step_at_the_partitions_edges(n_h, n_e):
    p = W.preset("track_200keV_320um")
    params = oracle.make_params(p["sensor"], W.field_switches(), p["mobility"])
    n = n_h + n_e
    xyz = W.random_cloud(n, 3.0, center=(1.0, -2.0, 160.0), seed=n)
    xyz[n_h:, 2] += 5.0
    sign = np.where(np.arange(n) < n_h, 1, -1).astype(np.int8)
    with cts.Simulator(p["sensor"], p["mobility"], max_slots=4) as sim:
        g_pos, g_st = cts.sim_debug_step(sim.h, 7, 3, xyz, sign)
    o_pos, o_st = oracle.step(params, 7, 3, 0, xyz.copy(), sign, np.zeros(n, dtype=np.int8))
    assert np.array_equal(g_st, o_st)
    d = o_pos - xyz
    rel = np.linalg.norm(g_pos - o_pos, axis=1) / np.linalg.norm(d, axis=1)
    # the bounds of the one-step parity tests (FP32 arithmetic of the step)
    assert np.median(rel) < 4e-7
    assert rel.max() < 2e-4


def test_small_events_run_to_the_end_beside_larger_ones():
    name = "plain_3keV_100um"
    p = W.preset(name)
    events = W.make_events(name, n=10, first_id=300)
    for ev, n in zip(events, (1, 2, 3, 5, 40, 64, 65, 200, 829, 1100)):
        ev["n_pairs"] = n
    with cts.Simulator(p["sensor"], p["mobility"], keep_final_xy=1) as sim:
        got = sim.run(events, keep_xy_capacity=1100)
        again = sim.run(events, keep_xy_capacity=1100)
    refs = oracle.run_events(oracle.make_params(p["sensor"], W.field_switches(), p["mobility"]),
                             events)
    for ev, g, a, r in zip(events, got, again, refs):
        assert g["status"] == r.status == 0
        assert g["n_collected"] == r.n_collected == ev["n_pairs"]
        assert abs(g["n_steps"] - r.n_steps) <= 1
        assert np.array_equal(g["pixels"], r.pixels)
        assert np.array_equal(g["pixels"], a["pixels"]) and g["n_steps"] == a["n_steps"]
        # the same bits every run, whatever the CTAs' timing
        assert np.array_equal(g["final_xy"], a["final_xy"])
        assert g["interactions"] == a["interactions"]
