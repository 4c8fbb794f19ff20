"""The work a user of the library has it do, as measurable cases.

A case is a beam on a phantom (or several) with a number of histories and a way
to read the result back; run() makes the calls a program makes through
paper_0910_0329_gb300.dpm.  Random numbers are keyed by (seed, history,
particle) and the tally is integer, so the same state gives the same outputs.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_0910_0329_gb300 import dpm
from paper_0910_0329_gb300 import workloads as W

PARAMS = dict(W.DEFAULT_PARAMS)
SIZES = [(64, 64, 64), (96, 96, 96), (128, 128, 128)]


def _beam(particle, energy, field, gantry=0.0):
    return {"particle": particle, "energy": energy, "field": field, "gantry": gantry}


E6MV = 0.0  # energy of a photon beam with the synthetic 6 MV spectrum


def _run(name, phantom, dims, d, beam, n, read, n_batches=0, refresh=False, count=False, sauter=False, dz=0.0):
    return {"name": name, "kind": "run", "phantom": phantom, "nx": dims[0], "ny": dims[1], "nz": dims[2], "d": d,
            "dz": dz or d, **beam, "n": n, "read": read, "n_batches": n_batches, "refresh": refresh, "count": count,
            "sauter": sauter}


def listed():
    return [
        # the smallest call: a 15 MeV photon pencil (pairs, positrons) on a ragged water phantom,
        # as a program probes a beam: launches and latency count
        _run("pencil-15MeV-2e3", "water", (21, 17, 40), 0.5, _beam("photon", 15.0, 0.2), 2000, "host"),
        # the small electron configuration: 20 MeV, 5x5 cm, water/lung/water, 2x10^4 histories
        _run("e20-slab-2e4", "wlw", (61, 61, 60), 0.5, _beam("electron", 20.0, 5.0), 20_000, "host"),
        # an electron field of a middle energy on an odd-sized patient-like phantom, with the event
        # counters and the stop rule's D_max query
        _run("e9-blob-count-3e5", "blob", (97, 83, 101), 0.31, _beam("electron", 9.0, 8.0), 300_000, "dmax",
             n_batches=20, count=True),
        # adaptive planning: the resident phantom's contents are replaced from host arrays, an oblique 6 MV
        # field of 10^6 histories is run, and dose and sigma stay on the device for the next stage
        _run("6mv-blob128-refresh-1e6", "blob", (128, 128, 128), 0.3, _beam("photon", E6MV, 10.0, 35.0), 1_000_000,
             "device", refresh=True),
        # 400 keV photons in bone with Sauter's photoelectron angles
        _run("sauter-400keV-2e6", "bone", (41, 41, 40), 0.25, _beam("photon", 0.4, 4.0), 2_000_000, "device",
             sauter=True),
        # the headline configuration: 6 MV, 10x10 cm, water/bone/water, 10^7 histories
        _run("6mv-slab-1e7", "wbw", (61, 61, 60), 0.5, _beam("photon", E6MV, 10.0), 10_000_000, "host"),
        # a long launch in the paper's geometry (0.2 cm slices, water/lung/water)
        _run("6mv-paper-5e7", "paper-lung", (61, 61, 150), 0.5, _beam("photon", E6MV, 10.0), 50_000_000, "device",
             dz=0.2),
        # the large electron configuration: 20 MeV on 128^3 blobs, 10^7 histories
        _run("e20-blob128-1e7", "blob", (128, 128, 128), 0.25, _beam("electron", 20.0, 10.0), 10_000_000, "device"),
        # transport into a caller's device tally without device allocation
        {"name": "noalloc-6mv-3e5", "kind": "noalloc", "phantom": "wbw", "nx": 61, "ny": 61, "nz": 60, "d": 0.5,
         "dz": 0.5, **_beam("photon", E6MV, 10.0), "n": 300_000},
        # eight phantoms and beams of uneven size in one graph-replayed batch
        {"name": "batch-8", "kind": "batch", "jobs": 8, "mix": 3, "n_lo": 5.0, "n_hi": 6.3, "graph": True},
        # one dose request to 1 % sigma at D_max: a 6 MV beamlet on a resident 128^3 phantom
        {"name": "serve-1", "kind": "serve", "requests": 1, "geometries": 1, "mix": 5, "target": 0.01},
        # six requests that share rounds, over two geometries
        {"name": "serve-6", "kind": "serve", "requests": 6, "geometries": 2, "mix": 6, "target": 0.01},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["run"] * 6 + ["noalloc", "batch", "serve"])
    if kind == "batch":
        return {"kind": kind, "jobs": rng.randint(3, 10), "mix": rng.randrange(1 << 20), "n_lo": 4.0, "n_hi": 6.0,
                "graph": rng.random() < 0.5}
    if kind == "serve":
        return {"kind": kind, "requests": rng.randint(1, 6), "geometries": rng.randint(1, 3),
                "mix": rng.randrange(1 << 20), "target": round(rng.uniform(0.01, 0.03), 4)}
    electron = rng.random() < 0.45
    if electron:
        e = round(rng.uniform(6.0, 20.0), 2)
        beam = _beam("electron", e, round(rng.uniform(3.0, 10.0), 2))
        n_max = 6e6 * 20.0 / e
    else:
        e = E6MV if rng.random() < 0.7 else round(rng.uniform(0.3, 15.0), 2)
        beam = _beam("photon", e, round(rng.uniform(0.2, 10.0), 2))
        n_max = 2e7
    beam["gantry"] = round(rng.uniform(-180.0, 180.0), 1) if rng.random() < 0.4 else 0.0
    dims = [_log(rng, 17, 140) for _ in range(3)]
    d = round(rng.uniform(0.2, 0.5), 3)
    if kind == "noalloc":
        return {"kind": kind, "phantom": rng.choice(["wlw", "wbw", "blob"]), "nx": dims[0], "ny": dims[1],
                "nz": dims[2], "d": d, "dz": d, **beam, "n": _log(rng, 1e3, n_max / 20)}
    c = _run("", rng.choice(["wlw", "wbw", "blob", "blob", "water"]), dims, d, beam, _log(rng, 1e3, n_max),
             rng.choice(["host", "device", "dmax"]), n_batches=rng.choice([0, 0, 10, 20]), refresh=rng.random() < 0.25,
             count=rng.random() < 0.2, sauter=not electron and rng.random() < 0.15)
    del c["name"]
    return c


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _phantom(kind, nx, ny, nz, d, dz, seed):
    if kind == "blob":
        return W.blob_phantom(nx, ny, nz, d, seed)
    if kind == "paper-lung":
        return W.paper_slab_phantom("lung")
    water, lung, bone = (W.MAT_WATER, 1.0), (W.MAT_LUNG, 0.3), (W.MAT_BONE, 1.85)
    slabs = {"water": [(0, 1e9, *water)], "bone": [(0, 1e9, *bone)],
             "wlw": [(0, 3, *water), (3, 10, *lung), (10, 1e9, *water)],
             "wbw": [(0, 3, *water), (3, 7, *bone), (7, 1e9, *water)]}[kind]
    return W.slab_phantom(nx, ny, nz, d, slabs)


def _source(c, ph):
    photon = c["particle"] == "photon"
    particle = W.PHOTON if photon else W.ELECTRON
    spectrum, energy = (W.SPEC_6MV, 6.0) if photon and c["energy"] == E6MV else (W.SPEC_MONO, c["energy"])
    if c["gantry"]:
        X, Y, Z = ph.extent
        return W.Source(particle, spectrum, energy, (X / 2, Y / 2, Z / 2), 100.0, c["field"], c["field"], c["gantry"])
    return W.axial_source(ph, particle, spectrum, energy, ssd=90.0, sad=100.0, fx=c["field"], fy=c["field"])


_session = None


def _shared():
    """The context that a program keeps for its runs: tables, queues and a stream."""
    global _session
    if _session is None:
        stream = torch.cuda.Stream()
        _session = dpm.Dpm(0, W.MATERIALS, PARAMS, stream=stream), stream
    return _session


class _State:
    def __init__(self, case):
        self.case, self.own, self.ctx, self.phantoms = case, None, None, []

    def __del__(self):
        try:
            if self.own is not None:
                self.own.close()
            else:
                for pid in self.phantoms:
                    dpm.dpm_free_phantom(self.ctx.ctx, pid)
        except Exception:
            pass


def prepare(case, seed):
    s = _State(case)
    if case["kind"] in ("run", "noalloc"):
        s.ctx, s.stream = _shared()
        ph = _phantom(case["phantom"], case["nx"], case["ny"], case["nz"], case["d"], case["dz"], seed)
        s.phantom, s.source, s.seed = ph, _source(case, ph), seed
        s.pid = s.ctx.load_phantom(ph)
        s.phantoms.append(s.pid)
        if case["kind"] == "noalloc":
            s.tally = torch.empty(ph.n_vox, dtype=torch.int64, device="cuda")
        else:
            s.opts = dict(n_batches=case["n_batches"], count_events=int(case["count"]),
                          physics_flags=dpm.SAUTER if case["sauter"] else 0)
            if case["read"] != "host":
                s.dose, s.sigma = (torch.empty(ph.n_vox, dtype=torch.float64, device="cuda") for _ in range(2))
        return s
    # a batch (its captured graph) and a server (its slots) belong to a context of their own
    s.ctx = s.own = dpm.Dpm(0, W.MATERIALS, PARAMS)
    g = W.SplitMix64(case["mix"])
    if case["kind"] == "batch":
        s.jobs, s.out = [], []
        for i in range(case["jobs"]):
            nx, ny, nz = SIZES[min(int(g.uniform() * 3), 2)]
            ph = W.blob_phantom(nx, ny, nz, round(0.2 + 0.3 * g.uniform(), 3), 64 * seed + i)
            if i % 2 == 0:
                src = W.axial_source(ph, W.PHOTON, W.SPEC_6MV, 6.0, ssd=90.0, sad=100.0, fx=10.0, fy=10.0)
            else:
                src = W.axial_source(ph, W.ELECTRON, W.SPEC_MONO, 6.0 + int(g.uniform() * 15), ssd=90.0, sad=100.0,
                                     fx=10.0, fy=10.0)
            n = int(round(10 ** (case["n_lo"] + (case["n_hi"] - case["n_lo"]) * g.uniform())))
            if i % 2:
                n = max(1, n // 8)
            s.jobs.append((s.ctx.load_phantom(ph), src, 0, n, 64 * seed + i))
            s.out.append(tuple(torch.empty(ph.n_vox, dtype=torch.float64, device="cuda") for _ in range(2)))
        return s
    geoms = [W.blob_phantom(128, 128, 128, 0.3, 16 * seed + k) for k in range(case["geometries"])]
    s.geoms = [s.ctx.load_phantom(ph) for ph in geoms]
    s.server = dpm.Server(s.ctx.ctx, dpm.serve_opts(target=case["target"]))
    s.requests = []
    for i in range(case["requests"]):
        k = int(g.uniform() * case["geometries"])
        X, Y, Z = geoms[k].extent
        src = W.Source(W.PHOTON, W.SPEC_6MV, 6.0, (X / 2, Y / 2, Z / 2), 100.0, 0.5, 0.5, 360.0 * g.uniform())
        s.requests.append((s.geoms[k], src, 1_000_000 + 64 * seed + i))
    s.dose, s.sigma = (torch.empty((case["requests"], geoms[0].n_vox), dtype=torch.float64, device="cuda")
                       for _ in range(2))
    return s


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------
def _summary(st, count=False):
    out = {k: st[k] for k in ("n_histories", "emitted", "deposited", "escaped", "missed", "error_flags")}
    if count:
        out.update({k: st[k] for k in ("n_e_steps", "n_g_flights", "n_g_interactions", "n_pushed")})
    return out


def run(s):
    c, d = s.case, s.ctx
    if c["kind"] == "run":
        if c["refresh"]:
            d.update_phantom(s.pid, s.phantom)
        else:
            d.reset(s.pid)
        d.run(s.pid, s.source, c["n"], s.seed, **s.opts)
        if c["read"] == "host":
            dose, sigma, raw, st = d.read(s.pid)
            return {"dose": dose, "sigma": sigma, "raw": raw, "stats": _summary(st, c["count"])}
        out = {}
        if c["read"] == "dmax":
            out["dmax"] = dpm.dpm_dmax_sigma(d.ctx, [s.pid])
        st = dpm.dpm_read_dose_device(d.ctx, s.pid, s.dose, s.sigma)
        return {"dose": s.dose, "sigma": s.sigma, "stats": _summary(st, c["count"]), **out}
    if c["kind"] == "noalloc":
        with torch.cuda.stream(s.stream):
            s.tally.zero_()
        st = dpm.dpm_run_noalloc(d.ctx, s.pid, s.source, 0, c["n"], s.seed, s.tally.data_ptr())
        st.pop("deposited")  # the tally's increase
        return {"tally": s.tally, "emitted": st["emitted"], "escaped": st["escaped"], "missed": st["missed"],
                "n_e_steps": st["n_e_steps"], "n_pushed": st["n_pushed"]}
    if c["kind"] == "batch":
        for job in s.jobs:
            d.reset(job[0])
        dpm.dpm_run_batch(d.ctx, s.jobs, dpm.run_opts(use_graph=int(c["graph"])))
        st = dpm.dpm_batch_stats(d.ctx)
        out = []
        for job, (dose, sigma) in zip(s.jobs, s.out):
            one = dpm.dpm_read_dose_device(d.ctx, job[0], dose, sigma)
            out.append({"dose": dose, "sigma": sigma, "deposited": one["deposited"]})
        return {"jobs": out, "emitted": st["emitted"], "escaped": st["escaped"], "missed": st["missed"]}
    ids = [s.server.submit(*r) for r in s.requests]
    while any(s.server.status(i)["state"] in (dpm.REQ_PENDING, dpm.REQ_ACTIVE) for i in ids):
        s.server.round()
    out = []
    for k, i in enumerate(ids):
        st = s.server.status(i)
        dpm.dpm_read_dose_device(d.ctx, st["slot"], s.dose[k], s.sigma[k])
        s.server.release(i)
        out.append({k2: st[k2] for k2 in ("histories", "rounds", "rel_sigma", "dose_max", "dmax_voxel")})
    return {"dose": s.dose, "sigma": s.sigma, "requests": out}


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------
def _history_flops(c):
    """Floating-point operations of one history: about 150 per condensed-history
    step (25 steps per MeV at these voxel sizes) and 40 per Woodcock flight."""
    if c["particle"] == "electron":
        return 25.0 * c["energy"] * 150.0
    mean = 1.7 if c["energy"] == E6MV else c["energy"]
    return 15.0 * 40.0 + 0.55 * 25.0 * mean * 150.0


def work(case):
    if case["kind"] in ("run", "noalloc"):
        vox = case["nx"] * case["ny"] * case["nz"]
        out = 8 if case["kind"] == "noalloc" else 24 if case["read"] == "host" else 16
        return {"bytes": vox * (5 + out), "flops": case["n"] * _history_flops(case)}
    if case["kind"] == "batch":
        g, b, f = W.SplitMix64(case["mix"]), 0, 0.0
        for i in range(case["jobs"]):
            nx, ny, nz = SIZES[min(int(g.uniform() * 3), 2)]
            g.uniform()
            e = 6.0 + int(g.uniform() * 15) if i % 2 else E6MV
            n = int(round(10 ** (case["n_lo"] + (case["n_hi"] - case["n_lo"]) * g.uniform())))
            beam = {"particle": "electron" if i % 2 else "photon", "energy": e}
            b += nx * ny * nz * 21
            f += (max(1, n // 8) if i % 2 else n) * _history_flops(beam)
        return {"bytes": b, "flops": f}
    # a 6 MV beamlet needs about 2x10^6 histories for 1 % sigma at D_max
    n = 2e6 * (0.01 / case["target"]) ** 2 * case["requests"]
    return {"bytes": 128 ** 3 * (5 * case["geometries"] + 16 * case["requests"]),
            "flops": n * _history_flops({"particle": "photon", "energy": E6MV})}


def exact(case, seed):
    """A Monte Carlo result has no closed form in 64 bits: its tally follows from
    the random numbers and the single-precision tracks, bit for bit."""
    return None
