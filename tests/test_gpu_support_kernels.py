"""The kernels around the steps where their split over CTAs has edges: events
whose carriers start collected, exited or reflected, empty and one-carrier
events beside larger ones, binning near pixel edges, and slots that are used
again by the next events."""
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


def test_start_states_match_the_oracle_and_slots_are_reused():
    # events at both surfaces: part of the cloud starts collected, exited or
    # reflected; two slots only, so that every slot serves several events
    p = W.preset("mip_50um")
    params = oracle.make_params(p["sensor"], W.field_switches(), p["mobility"])
    evs = [dict(seed=9, event_id=k, kind=W.PHOTON, energy_keV=1.0, n_pairs=n, depth_um=d, x_um=3.0,
                y_um=-4.0, sigma_um=2.0)
           for k, (n, d) in enumerate([(1, 0.0), (63, 0.0), (64, 50.0), (65, 25.0), (257, 49.0),
                                       (700, 1.0)])]
    with cts.Simulator(p["sensor"], p["mobility"], max_slots=2, keep_final_xy=1) as sim:
        got = sim.run(evs, keep_xy_capacity=1400)
        again = sim.run(evs, keep_xy_capacity=1400)
    refs = oracle.run_events(params, evs)
    for g, a, r in zip(got, again, refs):
        assert g["status"] == r.status == 0
        assert g["n_collected"] == r.n_collected and g["n_outside"] == r.n_outside
        assert g["pixels"].sum() + g["n_outside"] == g["n_collected"]
        start = g["retire_step"] == -1
        ref_start = np.asarray(r.retire_step)[:g["n_carriers"]] == -1
        assert np.array_equal(start, ref_start)
        assert np.array_equal(g["pixels"], a["pixels"])
        assert np.array_equal(g["retire_step"], a["retire_step"])


def test_an_empty_event_ends_at_once():
    p = W.preset("plain_3keV_100um")
    ev = W.make_events("plain_3keV_100um", n=2)
    empty = dict(ev[1], kind=W.EXPLICIT, explicit_xyz=np.zeros((0, 3)), n_pairs=0)
    with cts.Simulator(p["sensor"], p["mobility"]) as sim:
        got = sim.run([ev[0], empty])
    assert [g["status"] for g in got] == [0, 0]
    assert got[0]["n_collected"] == 829 and got[1]["n_collected"] == 0
    assert got[1]["pixels"].sum() == 0


@pytest.mark.parametrize("pitch,grid", [(25.0, 9), (55.0, 256), (0.3, 5)])
def test_binning_near_pixel_edges(pitch, grid):
    # points on, just below and just above pixel edges (FP64 spacing), where
    # FP32 must leave the decision to FP64, and points anywhere
    rng = np.random.default_rng(4)
    edge = (np.arange(-2, grid + 3) - 0.5 * grid) * pitch
    x = np.concatenate([edge, np.nextafter(edge, -1e9), np.nextafter(edge, 1e9),
                        edge * (1 + 1e-7), rng.uniform(-1.5, 1.5, 3000) * grid * pitch,
                        [0.0, 1e12, -1e12, 1e300]])
    y = rng.permutation(x)
    s = dict(W.preset("plain_3keV_100um")["sensor"], pitch_um=pitch, grid_n=grid)
    with cts.Simulator(s, W.preset("plain_3keV_100um")["mobility"]) as sim:
        pix, out = sim.bin(x, y)
    ix, iy = np.floor(x / pitch + 0.5 * grid), np.floor(y / pitch + 0.5 * grid)
    on = (ix >= 0) & (iy >= 0) & (ix < grid) & (iy < grid)
    ref = np.zeros((grid, grid), dtype=np.int64)
    np.add.at(ref, (iy[on].astype(int), ix[on].astype(int)), 1)
    assert np.array_equal(pix, ref) and out == (~on).sum()


def test_spherical_width_follows_the_running_events():
    # 40 events: two CTAs each while all run, four once few are left; the
    # same results as with one CTA throughout
    name = "plain_3keV_100um"
    p = W.preset(name)
    evs = W.make_events(name, n=40, first_id=10)
    outs = []
    for opt in ({}, dict(sph_cluster=1)):
        with cts.Simulator(p["sensor"], p["mobility"], W.field_switches(spherical=1),
                           keep_final_xy=1, **opt) as sim:
            outs.append(sim.run(evs, keep_xy_capacity=829))
            assert (sim.stats()["sph_cluster"] == 1) == bool(opt)
    for a, b in zip(*outs):
        assert a["n_steps"] == b["n_steps"] and np.array_equal(a["pixels"], b["pixels"])
        assert np.array_equal(a["final_xy"], b["final_xy"])
