"""Performance cases of the charge-transport library: what its users run.

Most time goes into simulating events (photons, minimum-ionising particles,
electron tracks) through ``Simulator.run``, from one small photon to a batch
that fills the GPU, with and without the recorded signals, by the pairwise
and by the spherical model.  Beside it stand the pair field for callers that
own their device buffers, the fast generation of events from the generalised
Gaussian model and the detector readout of pixel maps, both host to host.

What the cases return.  A simulated cloud is a chaotic N-body system: another
order of the FP32 sums moves single carriers by micrometres after a thousand
steps (and the FP64 oracle's run is no closer to either).  What a program
reads from it is not chaotic, and is what is compared: the charge per pixel
(beams aimed into a pixel, so that no carrier's side of a pixel border hangs
on a rounding), the counts of collected carriers, and the induced signals of
the electrodes, which sum over all carriers.  Step counts of single carriers,
the electrons still moving at the end and the work statistics are left out.  The library computes the signals from
FP32 fields; they are kept as float32, as a program that stores them does.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2506_09712_gb300 as cts
import workloads as W

# Bounds of the drawn cases.
FIELD_MIN, FIELD_MAX = 64, 131072    # carriers of cts_field_noalloc (its documented maximum)
COST_MAX = 1.4e12                    # ordered pair interactions of the largest listed case
EXACT_MAX = 1.6e11                   # ... up to which the 64-bit run stays under 20 seconds
# Steps after which a 64-bit run of the same chaotic system says nothing more:
# two FP32 runs in another order are as far from it as from each other.
EXACT_STEPS = 128


def listed():
    return [
        # the pair field on a caller's device buffers: the cloud of one 3 keV
        # photon, the smallest of the presets (launches and latency)
        dict(name="field_829", kind="field", n_h=829, n_e=0, sigma=1.0),
        # ... and one 200 keV track's holes and electrons, near the call's maximum
        dict(name="field_110500_both", kind="field", n_h=55250, n_e=55250, sigma=4.0),
        # one low-energy photon from start to readout: per-step latency
        dict(name="photon_3keV", kind="events", preset="plain_3keV_100um", n=1, e_lo=3.0,
             e_hi=3.0, pitch=25.0, steps=0, signals=0, spherical=0),
        # the 3 keV preset's eight photons in one call
        dict(name="batch_3keV_8", kind="events", preset="plain_3keV_100um", n=8, e_lo=3.0,
             e_hi=3.0, pitch=25.0, steps=0, signals=1, spherical=0),
        # one 20 keV photon with the collecting surface's signal: the few-event
        # regime, which also ends every batch
        dict(name="photon_20keV_signal", kind="events", preset="batch_20keV_320um", n=1,
             e_lo=20.0, e_hi=20.0, pitch=55.0, steps=0, signals=1, spherical=0),
        # the batch the library is benchmarked on: 64 photons of 20 keV
        dict(name="batch_20keV_64", kind="events", preset="batch_20keV_320um", n=64, e_lo=20.0,
             e_hi=20.0, pitch=55.0, steps=0, signals=0, spherical=0),
        # ten minimum-ionising particles, electrons and holes
        dict(name="mip_10", kind="tracks", preset="mip_50um", n=10, n_pairs=4000, pitch=25.0,
             steps=0, signals=1),
        # a 200 keV electron track's first steps: 110 500 carriers, the largest event
        dict(name="track_200keV", kind="tracks", preset="track_200keV_320um", n=1,
             n_pairs=55250, pitch=25.0, steps=12, signals=1),
        # the spherical comparison model on the batch
        dict(name="spherical_64", kind="events", preset="batch_20keV_320um", n=64, e_lo=20.0,
             e_hi=20.0, pitch=55.0, steps=0, signals=0, spherical=1),
        # transient pixel signals while the clouds drift
        dict(name="pixel_signals_8", kind="events", preset="serve_mix_320um", n=8, e_lo=5.0,
             e_hi=17.5, pitch=25.0, steps=64, signals=3, spherical=0),
        # fast generation: a few thousand events of the batch's energy per call
        dict(name="generate_5000", kind="generate", n=5000, n_pairs=5525, grid=9),
        # detector readout of as many pixel maps as an acquisition holds
        dict(name="readout_20000", kind="readout", n=20000, grid=9, pixels=0),
    ]


def _log_uniform(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["field", "field", "events", "events", "events", "events", "spherical",
                       "tracks", "pixels", "generate", "readout"])
    while True:
        if kind == "field":
            n = int(_log_uniform(rng, FIELD_MIN, FIELD_MAX))
            n_e = int(n * rng.uniform(0.2, 0.6)) if rng.random() < 0.4 else 0
            return dict(kind="field", n_h=n - n_e, n_e=n_e, sigma=rng.uniform(0.8, 5.0))
        if kind in ("events", "spherical", "pixels"):
            c = dict(kind="events", spherical=int(kind == "spherical"), steps=0, signals=0)
            if kind == "events" and rng.random() < 0.4:  # the 100 um sensor's energies
                c.update(preset="plain_3keV_100um", n=int(_log_uniform(rng, 1, 200)), pitch=25.0)
                c["e_lo"] = rng.uniform(2.0, 3.0)
                c["e_hi"] = rng.uniform(3.0, 4.0)
                c["signals"] = int(rng.random() < 0.3)
            else:
                c.update(preset=rng.choice(["batch_20keV_320um", "serve_mix_320um",
                                            "uneven_5_25keV_450um"]),
                         n=int(_log_uniform(rng, 1, 64)), pitch=55.0)
                if c["preset"] == "uneven_5_25keV_450um":
                    c["pitch"] = 75.0  # its clouds spread further
                c["e_lo"] = rng.uniform(5.0, 20.0)
                c["e_hi"] = min(25.0, c["e_lo"] * rng.uniform(1.0, 2.5))
                c["signals"] = int(rng.random() < 0.3)
            if kind == "pixels":
                c.update(n=int(_log_uniform(rng, 1, 16)), signals=3, steps=rng.randint(32, 72),
                         pitch=25.0)
        elif kind == "tracks":
            if rng.random() < 0.5:
                c = dict(kind="tracks", preset="mip_50um", n=int(_log_uniform(rng, 1, 16)),
                         n_pairs=rng.randint(2000, 6000), pitch=25.0, steps=0, signals=1)
            else:
                c = dict(kind="tracks", preset="track_200keV_320um", n=rng.randint(1, 4),
                         n_pairs=int(_log_uniform(rng, 8000, 55250)), pitch=25.0,
                         steps=rng.randint(6, 14), signals=1)
        elif kind == "generate":
            return dict(kind="generate", n=int(_log_uniform(rng, 10, 10000)),
                        n_pairs=rng.randint(800, 7000), grid=rng.choice([5, 9, 17]))
        else:
            return dict(kind="readout", n=int(_log_uniform(rng, 10, 40000)),
                        grid=rng.choice([5, 9, 17]), pixels=int(rng.random() < 0.3))
        if _interactions(c) <= (20.0 if c.get("spherical") else 1.0) * COST_MAX:
            return c


# ---- what a case's events are --------------------------------------------------
def _preset(case):
    p = W.preset(case["preset"])
    p["sensor"]["pitch_um"] = case["pitch"]
    if case["steps"]:
        p["sensor"]["max_steps"] = case["steps"]
    return p


def _events(case, seed):
    """Descriptors made from the seed: depths by the workload's absorption
    law, entry points near the middle of the grid's centre pixel: a beam
    focused into it (narrower where the clouds grow wider)."""
    p = _preset(case)
    rng = np.random.default_rng([seed, 0xCA5E])
    n, s = case["n"], p["sensor"]
    wide = 0.05 if case["pitch"] > 50.0 else 0.15
    xy = rng.uniform(-wide, wide, (n, 2)) * s["pitch_um"]
    base = dict(seed=int(rng.integers(1 << 48)), sigma_um=p["sigma_um"])
    ids = int(rng.integers(1 << 20))
    out = []
    if case["kind"] == "tracks":
        theta, phi = rng.uniform(0.0, p["theta_max_deg"], n), rng.uniform(0.0, 360.0, n)
        for k in range(n):
            out.append(dict(base, event_id=ids + k, kind=W.TRACK, energy_keV=200.0,
                            n_pairs=case["n_pairs"], x_um=float(xy[k, 0]), y_um=float(xy[k, 1]),
                            track_len_um=p["track_len_um"], theta_deg=float(theta[k]),
                            phi_deg=float(phi[k])))
        return p, out
    energy = rng.uniform(case["e_lo"], case["e_hi"], n)
    # one draw per event keeps the sets of energies and depths independent
    depth = np.array([W.sample_depths(rng, e, s["thickness_um"])[0] for e in energy])
    for k in range(n):
        out.append(dict(base, event_id=ids + k, kind=W.PHOTON, energy_keV=float(energy[k]),
                        n_pairs=int(round(energy[k] * 1000.0 / 3.62)), x_um=float(xy[k, 0]),
                        y_um=float(xy[k, 1]), depth_um=float(depth[k])))
    return p, out


def _steps(case):
    """Steps that the events of a case take on average: their number, or the
    drift time from a mean depth through the sensor."""
    p = _preset(case)
    s, m = p["sensor"], p["mobility"]
    H, steps, z, dt = s["thickness_um"], 0, 0.0, s["dt_ps"] * 1e-3
    z = H if case["kind"] == "tracks" else 0.6 * H
    dz = H / 400.0
    t = 0.0
    while z > 0.0:
        E = (s["bias_V"] + s["depletion_V"]) / H - 2.0 * s["depletion_V"] * z / H**2
        mu0, vs, be = m["mu0_h"] * 0.1, m["vsat_h"] * 1e-5, m["beta_h"]
        t += dz / (mu0 * E / (1.0 + (mu0 * E / vs) ** be) ** (1.0 / be))
        z -= dz
    steps = int(t / dt) + 1
    return min(steps, case["steps"]) if case["steps"] else steps


def _carriers(case):
    """(holes and electrons of an event on average, mean square)."""
    if case["kind"] == "tracks":
        return 2.0 * case["n_pairs"], 4.0 * case["n_pairs"] ** 2
    lo, hi = case["e_lo"] * 1000 / 3.62, case["e_hi"] * 1000 / 3.62
    return 0.5 * (lo + hi), (lo * lo + lo * hi + hi * hi) / 3.0


def _interactions(case):
    return case["n"] * _carriers(case)[1] * _steps(case)


# ---- the library's calls ---------------------------------------------------------
def prepare(case, seed):
    if case["kind"] == "field":
        g = torch.Generator(device="cuda").manual_seed(seed)
        n = case["n_h"] + case["n_e"]
        xyz = torch.randn(3, n, device="cuda", generator=g) * case["sigma"]
        xyz[2, case["n_h"]:] += 0.8  # the electrons' cloud has drifted away a little
        return dict(case=case, xyz=xyz.contiguous(), out=torch.empty(3, n, device="cuda"))
    if case["kind"] in ("events", "tracks"):
        p, events = _events(case, seed)
        field = W.field_switches(spherical=case.get("spherical", 0))
        sim = cts.Simulator(p["sensor"], p["mobility"], field, keep_induced=case["signals"],
                            keep_final_xy=case.get("spherical", 0))
        # room for every step of the longest drift, and the end of the record held
        cap = case["steps"] or 2 * _steps(case)
        carriers = int(case["e_hi"] * 1000.0 / 3.62) + 1 if case["kind"] == "events" else 0
        return dict(case=case, sim=sim, events=events, cap=cap, carriers=carriers)
    rng = np.random.default_rng([seed, 0xCA5E])
    n = case["n"]
    if case["kind"] == "generate":
        rec = cts.gen_events(int(rng.integers(1 << 48)), np.arange(n), case["n_pairs"],
                             rng.uniform(-12.5, 12.5, n), rng.uniform(-12.5, 12.5, n),
                             rng.uniform(3.0, 12.0, n), rng.uniform(2.0, 3.0, n))
        return dict(case=case, rec=rec)
    return dict(case=case, counts=_counts(rng, n, case["grid"]),
                seeds=rng.integers(1 << 62, size=n).astype(np.uint64),
                ids=np.arange(n, dtype=np.uint64))


def _counts(rng, n, grid):
    """Pixel maps of 20 keV clouds a few micrometres wide at any point of the
    centre pixel, and every tenth a second photon's elsewhere (pile-up)."""
    edges = (np.arange(grid + 1) - 0.5 * grid) * 25.0
    maps = np.zeros((n, grid, grid))
    for second in (0, 1):
        c = rng.uniform(-12.5, 12.5, (n, 2)) + second * rng.uniform(-50.0, 50.0, (n, 2))
        w = rng.uniform(3.0, 7.0, (n, 1))
        px = np.diff(np.tanh((edges - c[:, :1]) / w) * 0.5, axis=1)
        py = np.diff(np.tanh((edges - c[:, 1:]) / w) * 0.5, axis=1)
        on = 1.0 if second == 0 else (rng.random(n) < 0.1)[:, None, None]
        maps += 5525.0 * on * py[:, :, None] * px[:, None, :]
    return np.round(maps).astype(np.int32)


def run(state):
    case = state["case"]
    if case["kind"] == "field":
        xyz, out = state["xyz"], state["out"]
        rc = cts.cts_field_noalloc(xyz[0].data_ptr(), xyz[1].data_ptr(), xyz[2].data_ptr(),
                                   case["n_h"], case["n_e"], 11.7, 1e-6, out.data_ptr(),
                                   torch.cuda.current_stream().cuda_stream)
        if rc != cts.SIM_OK:
            raise cts.SimError(rc, "cts_field_noalloc")
        return out
    if case["kind"] == "generate":
        pixels, outside = cts.sim_generate(state["rec"], 25.0, case["grid"])
        return dict(pixels=pixels, outside=outside)
    if case["kind"] == "readout":
        r = cts.sim_readout(state["counts"], state["seeds"], state["ids"], 20.0, n_bins=300,
                            want_pixels=bool(case["pixels"]))
        return {k: r[k] for k in ("cluster", "e_cluster", "accepted", "vetoed", "cx", "cy",
                                  "spectrum", "e") if k in r}
    signals = case["signals"]
    rec = state["sim"].run(state["events"],
                           keep_xy_capacity=state["carriers"] if case.get("spherical") else 0,
                           induced_capacity=state["cap"] if signals else 0)
    out = {k: np.array([r[k] for r in rec], dtype=np.int64)
           for k in ("status", "n_collected", "n_outside")}
    out["pixels"] = np.stack([r["pixels"] for r in rec])
    if signals & 1:
        out["induced"] = _record([r["induced"] for r in rec], state["cap"], ())
    if signals & 2:
        out["induced_px"] = _record([r["induced_px"] for r in rec], state["cap"], (3, 3))
    if case.get("spherical"):
        # the spherical field is smooth: the collection points are comparable
        out["final_xy"] = np.zeros((len(rec), state["carriers"], 2), dtype=np.float32)
        for k, r in enumerate(rec):
            out["final_xy"][k, :len(r["final_xy"])] = r["final_xy"]
    return out


def _record(rows, cap, tail):
    """The events' charge signals as one float32 array, each held at its end
    value once its event is over."""
    out = np.zeros((len(rows), cap) + tail, dtype=np.float32)
    for k, v in enumerate(rows):
        m = min(len(v), cap)
        out[k, :m] = v[:m]
        if m:
            out[k, m:] = v[m - 1]
    return out


def work(case):
    if case["kind"] == "field":
        n = case["n_h"] + case["n_e"]
        # 22 flops per unordered pair (3 differences, 5 for r^2, 2 for r^-3
        # beside the rsqrt, 3 multiply-adds into each carrier's sum)
        return dict(bytes=24.0 * n, flops=11.0 * n * (n - 1.0))
    if case["kind"] == "generate":
        # four Philox blocks and two gamma variates a carrier, about 300 operations
        return dict(bytes=case["n"] * (56.0 + 8.0 + 4.0 * case["grid"] ** 2),
                    flops=300.0 * case["n"] * case["n_pairs"])
    if case["kind"] == "readout":
        g2 = case["grid"] ** 2
        return dict(bytes=case["n"] * (16.0 + 4.0 * g2 + 96.0 + 8.0 * g2 * case["pixels"]),
                    flops=150.0 * case["n"] * g2)
    n, steps = case["n"] * _carriers(case)[0], _steps(case)
    out = case["n"] * (4.0 * 81 + 64.0) + 8.0 * n  # maps, counts, drawn starts
    if case["signals"]:
        out += case["n"] * 4.0 * steps * (1 + 9 * (case["signals"] >> 1))
    update = n * steps * 120.0
    if case["signals"] & 2:
        update += n * steps * 80.0 * 30.0  # 5 image planes of 16 corner terms
    pairs = n * steps * 20.0 if case.get("spherical") else 11.0 * _interactions(case)
    return dict(bytes=out, flops=pairs + update)


# ---- the same in 64 bits, from the method's equations ------------------------------
def exact(case, seed):
    if case["kind"] == "field":
        s = prepare(case, seed)
        q = torch.ones(s["xyz"].shape[1], dtype=torch.float64, device="cuda")
        q[case["n_h"]:] = -1.0
        return _pair_field(s["xyz"].double(), q, _coulomb(11.7), 1e-12)
    if case["kind"] == "generate":
        return None  # whole numbers
    if case["kind"] == "readout":
        return _exact_readout(case, seed)
    if case.get("spherical") or not case["signals"] or _interactions(case) > EXACT_MAX or \
            _steps(case) > EXACT_STEPS:
        return None  # whole numbers, a run of over 20 seconds, or past the horizon
    return _exact_events(case, seed)


def _coulomb(eps_r):
    return 1.602176634e-19 / (4.0 * math.pi * 8.8541878128e-12 * eps_r) * 1e6


def _pair_field(r, q, kc, eps2):
    """Eq. 4: the field (3, n) of charges q at r (3, n)."""
    n = r.shape[1]
    out = torch.empty_like(r)
    rows = max(1, int(2.5e8 // max(n, 1)))
    for a in range(0, n, rows):
        d = [r[c, a:a + rows, None] - r[c, None, :] for c in range(3)]
        w = (d[0] * d[0]).addcmul_(d[1], d[1]).addcmul_(d[2], d[2]).add_(eps2)
        w = w.rsqrt_().pow_(3).mul_(q)
        for c in range(3):
            out[c, a:a + rows] = torch.einsum("ij,ij->i", d[c], w)
    return out * kc


def _philox(seed, event, purpose, carrier, step):
    """Philox4x32-10 words (4, n) of (carrier, step, event, purpose), key = seed."""
    u = np.uint64
    lo = u(0xFFFFFFFF)
    carrier, step = np.broadcast_arrays(np.asarray(carrier, u), np.asarray(step, u))
    event, seed = np.asarray(event, u), np.asarray(seed, u)
    c = [carrier.copy(), step.copy(), np.broadcast_to(event & lo, carrier.shape).copy(),
         np.broadcast_to((event >> u(32)) ^ u(purpose << 28), carrier.shape).copy()]
    k0, k1 = seed & lo, seed >> u(32)
    for _ in range(10):
        a, b = u(0xD2511F53) * c[0], u(0xCD9E8D57) * c[2]
        c = [(b >> u(32)) ^ c[1] ^ k0, b & lo, (a >> u(32)) ^ c[3] ^ k1, a & lo]
        k0, k1 = (k0 + u(0x9E3779B9)) & lo, (k1 + u(0xBB67AE85)) & lo
    return c


def _normals(w):
    un = [((x >> np.uint64(9)).astype(np.float64) + 0.5) * 2.0**-23 for x in w]
    r01, r23 = np.sqrt(-2.0 * np.log(un[0])), np.sqrt(-2.0 * np.log(un[2]))
    a, b = 2.0 * np.pi * un[1], 2.0 * np.pi * un[3]
    return np.stack([r01 * np.cos(a), r01 * np.sin(a), r23 * np.cos(b)])


def _exact_readout(case, seed):
    s = prepare(case, seed)
    n, g = case["n"], case["grid"]
    pix = np.arange(g * g, dtype=np.uint64)[None, :]
    w = _philox(s["seeds"][:, None], s["ids"][:, None], 3, np.broadcast_to(pix, (n, g * g)), 0)
    e = s["counts"].reshape(n, -1) * 3.62 * 1e-3 + 0.13 * _normals(w)[0]
    best = e.argmax(axis=1)
    pad = np.full((n, g + 2, g + 2), np.nan)
    pad[:, 1:-1, 1:-1] = e.reshape(n, g, g)
    cy, cx = best // g, best % g
    cl = np.stack([pad[np.arange(n), cy + dy, cx + dx] for dy in range(3) for dx in range(3)], 1)
    out = dict(cluster=cl, e_cluster=np.nansum(cl, axis=1))
    if case["pixels"]:
        out["e"] = e.reshape(n, g, g)
    return dict({k: None for k in ("accepted", "vetoed", "cx", "cy", "spectrum")}, **out)


def _window_potentials(r, s):
    """Weighting potentials (9, n) of the 3 x 3 pixels around the grid's
    centre at r (3, n): image pairs of the pixels' solid angles, the rest of
    the series by its two leading terms."""
    H, p, gn, M = s["thickness_um"], s["pitch_um"], s["grid_n"], 8
    c = gn // 2
    x0 = ((c - 1) - 0.5 * gn) * p
    u = [x0 + i * p - r[0] for i in range(4)]
    v = [x0 + i * p - r[1] for i in range(4)]
    F = torch.zeros((4, 4) + r[0].shape, dtype=torch.float64, device=r.device)
    for k in range(-M, M + 1):
        zeta = r[2] + 2.0 * k * H
        for j in range(4):
            for i in range(4):
                F[j, i] += torch.sign(zeta) * torch.atan2(
                    u[i] * v[j], zeta.abs() * (u[i]**2 + v[j]**2 + zeta**2).sqrt())
    s3 = 1.2020569031595942854 - sum(1.0 / k**3 for k in range(1, M + 1))
    s5 = 1.0369277551433699263 - sum(1.0 / k**5 for k in range(1, M + 1))
    w = (F[1:, 1:] - F[1:, :-1] - F[:-1, 1:] + F[:-1, :-1]) / (2.0 * math.pi)
    mid = [[0.5 * (a[i] + a[i + 1]) for i in range(3)] for a in (u, v)]
    far = torch.stack([torch.stack([cx**2 + cy**2 for cx in mid[0]]) for cy in mid[1]])
    w -= p * p * r[2] * (s3 / (4.0 * math.pi * H**3) - s5 / (16.0 * math.pi * H**5)
                         * (3.0 * (far + p * p / 6.0) - 2.0 * r[2]**2))
    w = w.reshape(9, -1)
    ix = torch.floor(r[0] / p + 0.5 * gn) - (c - 1)
    iy = torch.floor(r[1] / p + 0.5 * gn) - (c - 1)
    key = torch.where((ix >= 0) & (ix < 3) & (iy >= 0) & (iy < 3), iy * 3 + ix, -1.0)
    on = (key[None, :] == torch.arange(9, device=r.device)[:, None]).double()
    return torch.where(r[2] <= 0.0, on, torch.where(r[2] >= H, torch.zeros_like(w), w))


def _exact_events(case, seed):
    p, events = _events(case, seed)
    cap = case["steps"] or 2 * _steps(case)
    rows = [_exact_event(p, ev, cap, case["signals"]) for ev in events]
    out = {k: None for k in ("status", "n_collected", "n_outside", "pixels")}
    out["induced"] = torch.stack([r[0] for r in rows])
    if case["signals"] & 2:
        out["induced_px"] = torch.stack([r[1].reshape(-1, 3, 3) for r in rows])
    return out


def _exact_event(p, ev, cap, signals):
    """Algorithm 1 for one event: the induced charge after each step."""
    s, m = p["sensor"], p["mobility"]
    H, dt, kT = s["thickness_um"], s["dt_ps"] * 1e-3, 1.380649e-23 * s["temperature_K"] / 1.602176634e-19
    both, n = s["species"] == W.BOTH, ev["n_pairs"]
    ids = np.arange(n)
    g = _normals(_philox(ev["seed"], ev["event_id"], 1, ids, 0))
    sigma = ev["sigma_um"] if ev["sigma_um"] >= 0 else 0.0044 * ev["energy_keV"] ** 1.75
    if ev["kind"] == W.TRACK:
        th, ph = np.radians(ev["theta_deg"]), np.radians(ev["phi_deg"])
        w = _philox(ev["seed"], ev["event_id"], 1, ids, 1)[0]
        t = ((w >> np.uint64(9)).astype(np.float64) + 0.5) * 2.0**-23 * ev["track_len_um"]
        r = np.stack([ev["x_um"] + t * np.sin(th) * np.cos(ph)
                      + sigma * (g[0] * np.cos(th) * np.cos(ph) - g[1] * np.sin(ph)),
                      ev["y_um"] + t * np.sin(th) * np.sin(ph)
                      + sigma * (g[0] * np.cos(th) * np.sin(ph) + g[1] * np.cos(ph)),
                      H - t * np.cos(th) + sigma * g[0] * np.sin(th)])
    else:
        r = np.stack([ev["x_um"] + sigma * g[0], ev["y_um"] + sigma * g[1],
                      H - ev["depth_um"] + sigma * g[2]])
    if both:
        r, ids = np.concatenate([r, r], axis=1), np.arange(2 * n)
    q = np.where(ids < n, 1.0, -1.0)
    dev = dict(dtype=torch.float64, device="cuda")
    r, q = torch.tensor(r, **dev), torch.tensor(q, **dev)

    def bounds(r, q):
        """What leaves, and what is reflected at the other surface."""
        gone = torch.where(q > 0, r[2] <= 0.0, r[2] >= H)
        z = torch.where(q > 0, torch.where(r[2] > H, 2.0 * H - r[2], r[2]), torch.where(
            gone, r[2], r[2].abs()))
        return gone, torch.stack([r[0], r[1], z])

    gone, r = bounds(r, q)
    keep = ~gone
    r, q, ids = r[:, keep], q[keep], ids[keep.cpu().numpy()]
    total, px = torch.zeros(cap, **dev), torch.zeros(cap, 9, **dev)
    mob = [torch.tensor([m.get(k + "_h", 0.0), m.get(k + "_e", 0.0) or m[k + "_h"]], **dev)
           for k in ("mu0", "vsat", "beta")]
    phi = _window_potentials(r, s) if signals & 2 else None
    done = 0
    for step in range(cap):
        if not bool((q > 0).any()):
            break
        E = _pair_field(r, q, _coulomb(s["eps_r"]), s["softening_um"] ** 2)
        E[2] -= (s["bias_V"] + s["depletion_V"]) / H - 2.0 * s["depletion_V"] * r[2] / H**2
        sp = (q < 0).long()
        mu0, vs, be = mob[0][sp] * 0.1, mob[1][sp] * 1e-5, mob[2][sp]
        mu = mu0 / (1.0 + (mu0 * E.norm(dim=0) / vs) ** be) ** (1.0 / be)
        nrm = torch.tensor(_normals(_philox(ev["seed"], ev["event_id"], 0, ids, step)), **dev)
        new = r + q * mu * dt * E + (2.0 * mu * kT * dt).sqrt() * nrm
        gone, new = bounds(new, q)
        end = torch.stack([new[0], new[1], new[2].clamp(0.0, H)])
        last = total[step - 1] if step else 0.0
        total[step] = last + (q * (r[2] - end[2])).sum() / H
        if signals & 2:
            phi_new = _window_potentials(end, s)
            px[step] = (px[step - 1] if step else 0.0) + (q * (phi_new - phi)).sum(dim=1)
            phi = phi_new[:, ~gone]
        keep = ~gone
        r, q, ids = new[:, keep], q[keep], ids[keep.cpu().numpy()]
        done = step + 1
    if 0 < done < cap:
        total[done:], px[done:] = total[done - 1], px[done - 1]
    return total, px
