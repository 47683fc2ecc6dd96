"""The work that users of this library have it do, as measured cases.

A case names a scene, a set of seeded tracks (or photons) and the public call
that takes them through the library: the emit + trace step on device buffers,
its CUDA-graph replay, the host-to-host step, the gradient, the emission of
photon vectors and the trace of a caller's photons. Sizes are those of the
repository's workloads, tests and benchmark, or generic.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_2309_12496_gb300 import rich
from paper_2309_12496_gb300 import workloads as W

DEV = "cuda:0"

# scene -> (builder, n - 1, lambda range, mean photons per track, detected share,
#           surfaces met per photon, surfaces in the scene)
_SCENES = {
    "point": (lambda: W.point_source_scene(), 0.0014, (200.0, 600.0), 1.0, 0.12, 2.0, 2),
    "rich1": (lambda: W.rich1_scene(meshed=True), 0.0014, (200.0, 600.0), 350.0, 0.145, 2.7, 9),
    "rich1_analytic": (lambda: W.rich1_scene(meshed=False), 0.0014, (200.0, 600.0), 350.0, 0.145,
                       2.7, 9),
    "rich1_windows": (lambda: W.rich1_scene(meshed=True, windows=True), 0.0014, (200.0, 600.0),
                      350.0, 0.145, 4.2, 13),
    "rich2": (lambda: W.rich2_scene(meshed=True), 0.0005, (200.0, 600.0), 205.0, 0.13, 2.7, 61),
    "scint": (lambda: W.scint_box_scene(), 0.0, (350.0, 650.0), 2000.0, 0.295, 2.6, 6),
    "water": (lambda: W.water_tank_scene(), 0.33, (300.0, 600.0), 66000.0, 0.287, 1.0, 6),
}


@functools.lru_cache(maxsize=None)
def _scene(name):
    return _SCENES[name][0]()


def listed():
    return [
        # a calibration point source (the paper's ring test): one emitter, analytic mirror
        {"name": "point_100k", "kind": "step", "scene": "point", "tracks": 1, "photons": 100000,
         "events": 1, "precision": "refined", "fate": True},
        # one collision event through the synchronous host call: an online consumer, latency
        {"name": "event_host", "kind": "host", "scene": "rich1", "tracks": 47, "events": 1,
         "precision": "refined", "in_flight": 1},
        # the benchmark's step: 1000 tracks, meshed mirrors, device buffers
        {"name": "rich1_1000", "kind": "step", "scene": "rich1", "tracks": 1000, "events": 1,
         "precision": "refined"},
        # a stream of track batches from host memory, two steps in flight
        {"name": "stream_host", "kind": "host", "scene": "rich1", "tracks": 1013, "events": 20,
         "precision": "refined", "in_flight": 2},
        # reconstruction input: the hit list grouped by track for ring fits
        {"name": "ring_hits_10k", "kind": "step", "scene": "rich1", "tracks": 10007, "events": 1,
         "precision": "refined", "hits": True},
        # simulation of a run: many events of uneven size, one graph replay, counts per event
        {"name": "batch_graph", "kind": "graph", "scene": "rich1", "tracks": 25600, "events": 512,
         "precision": "refined"},
        # alignment: loss and gradient in mirror tilts, radius and index
        {"name": "gradient", "kind": "grad", "scene": "rich1_analytic", "tracks": 200,
         "photons": 5000, "events": 1, "precision": "refined"},
        # the large detector, a chunk of a long production
        {"name": "rich2_chunk", "kind": "step", "scene": "rich2", "tracks": 120011, "events": 1,
         "precision": "refined"},
        # scintillation light in a mirror box: many bounces on flat analytic walls
        {"name": "scint_box", "kind": "step", "scene": "scint", "tracks": 1999, "events": 1,
         "precision": "refined"},
        # wavelength-resolved radiator and quartz windows, with every photon's fate
        {"name": "dispersive_windows", "kind": "step", "scene": "rich1_windows", "tracks": 3001,
         "events": 1, "precision": "refined", "dispersive": True, "fate": True},
        # photons of another simulation handed in as vectors, FP32 positions
        {"name": "caller_photons", "kind": "external", "scene": "rich1", "tracks": 2000,
         "photons": 500, "events": 8, "precision": "fp32", "fate": True},
        # photon vectors handed out to another program
        {"name": "photon_vectors", "kind": "vectors", "scene": "rich1", "tracks": 2003,
         "events": 1, "precision": "refined"},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "host", "graph", "grad", "external", "vectors"])
    case = {"kind": kind, "precision": rng.choice(["refined", "refined", "fp32"])}
    if kind == "step":
        scene = rng.choice(["point", "rich1", "rich1", "rich1_analytic", "rich1_windows", "rich2",
                            "scint", "water"])
        hi = {"point": 1, "rich1": 30000, "rich1_analytic": 30000, "rich1_windows": 10000,
              "rich2": 100000, "scint": 3000, "water": 150}[scene]
        case.update(scene=scene, tracks=_log_int(rng, 1 if hi < 1000 else 10, hi), events=1)
        if scene == "point":
            case["photons"] = _log_int(rng, 1000, 1000000)
        if scene in ("rich1", "rich2"):
            case["prefilter"] = rng.random() < 0.25
            case["hits"] = rng.random() < 0.25
        if scene in ("rich1", "rich1_windows"):
            case["dispersive"] = rng.random() < 0.4
        case["fate"] = rng.random() < 0.4
    elif kind == "host":
        case.update(scene="rich1", tracks=_log_int(rng, 1, 5000), events=rng.randint(1, 30),
                    in_flight=rng.choice([1, 2]))
    elif kind == "graph":
        events = _log_int(rng, 4, 500)
        case.update(scene="rich1", events=events, tracks=events * rng.randint(20, 60) + 1)
    elif kind == "grad":
        case.update(scene="rich1_analytic", precision="refined", events=1,
                    tracks=_log_int(rng, 4, 400), photons=_log_int(rng, 100, 5000))
    elif kind == "external":
        case.update(scene=rng.choice(["rich1", "rich2"]), tracks=_log_int(rng, 2, 5000),
                    photons=rng.randint(30, 700), events=rng.randint(1, 40),
                    prefilter=rng.random() < 0.25, fate=True)
    else:
        case.update(scene="rich1", precision="refined", events=1, tracks=_log_int(rng, 2, 20000))
    return case


# ------------------------------------------------------------------- inputs
def _tracks(case, seed):
    scene, n, k = case["scene"], case["tracks"], case.get("photons")
    if scene == "point":
        return W.point_source_tracks(k)
    if scene == "scint":
        t = W.scint_tracks(n, seed=seed)
    elif scene == "water":
        t = W.water_muons(n, seed=seed)
    elif scene == "rich2":
        t = W.pion_tracks(n, seed=seed, length=2000.0, max_angle=0.15)
    elif case["kind"] == "grad":
        t = W.pion_tracks(n, seed=seed, n_fixed=k, p_min=3.0)
    else:
        t = W.pion_tracks(n, seed=seed)
    if case["events"] > 1:
        # uneven events: every track falls in one of them, ids count within it
        rng = np.random.default_rng([seed, 7])
        t.event = np.sort(rng.integers(0, case["events"], n)).astype(np.uint32)
        first = np.searchsorted(t.event, t.event)
        t.id = (np.arange(n) - first).astype(np.uint32)
    return t


def _capacity(case):
    """Photons that the buffers of a case hold: the yield is at most 1.5
    times the mean (momenta near threshold emit less)."""
    k = case.get("photons")
    return case["tracks"] * k if k else int(1.6 * case["tracks"] * _SCENES[case["scene"]][3]) + 1000


def _emission(case):
    _, n1, (l0, l1), *_ = _SCENES[case["scene"]]
    kw = dict(lambda_min=l0, lambda_max=l1)
    if case["scene"] == "scint":
        kw.update(source=rich.SOURCE_ISOTROPIC, yield_per_mm=20.0, spectrum_table=2)
    if case.get("dispersive"):
        kw["dispersion"] = W.C4F10_DISPERSION
    return n1, kw


def _trace_options(case):
    kw = dict(precision=rich.PREC_FP32 if case["precision"] == "fp32" else rich.PREC_REFINE64)
    if case.get("prefilter"):
        kw["prefilter"] = (0, 1, 2)          # QE, spherical and flat mirror reflectivity
    return kw


def _photon_vectors(case, seed):
    """Photons of tracks as another simulation would hand them in: origins
    along the track, directions on the Cherenkov cone, wavelengths of the
    1/lambda^2 spectrum, in track order."""
    g = torch.Generator(device=DEV).manual_seed(seed)
    t = _tracks(case, seed)
    per, n1 = case["photons"], _SCENES[case["scene"]][1]
    n = t.n * per

    def rep(a, dtype=torch.float64):
        return torch.from_numpy(np.asarray(a).astype(np.int64 if dtype == torch.int64
                                                     else np.float64)).to(DEV).repeat_interleave(per)

    def uniform():
        return torch.rand(n, generator=g, device=DEV, dtype=torch.float64)

    d = torch.stack([rep(t.dx), rep(t.dy), rep(t.dz)], 1)
    d = d / d.norm(dim=1, keepdim=True)
    p, m = rep(t.p), rep(t.mass)
    nb = ((1.0 + n1) * p / torch.sqrt(p * p + m * m)).clamp(min=1.0 + 1e-6)
    ct = 1.0 / nb
    st = torch.sqrt(1.0 - ct * ct)
    e1, e2 = _basis(d)
    phi = 2.0 * math.pi * uniform()
    dirs = d * ct[:, None] + (e1 * torch.cos(phi)[:, None] + e2 * torch.sin(phi)[:, None]) * st[:, None]
    o = torch.stack([rep(t.x), rep(t.y), rep(t.z)], 1) + d * (uniform() * rep(t.length))[:, None]
    l0, l1 = _SCENES[case["scene"]][2]
    lam = 1.0 / (1.0 / l0 - uniform() * (1.0 / l0 - 1.0 / l1))
    pb = rich.PhotonBuffers(n, DEV)
    for k, name in enumerate("xyz"):
        pb.t[name].copy_(o[:, k])
        pb.t["d" + name].copy_(dirs[:, k])
    pb.t["lambda_"].copy_(lam)
    pb.t["event"].copy_(rep(t.event, torch.int64))
    pb.t["track"].copy_(rep(t.id, torch.int64))
    pb.t["photon"].copy_(torch.arange(per, device=DEV).repeat(t.n))
    pb.n = n
    return pb


def _theta(case, seed):
    th = W.nominal_theta(_scene(case["scene"]), _SCENES[case["scene"]][1])
    rng = np.random.default_rng([seed, 11])
    th[:8] = rng.uniform(-2e-3, 2e-3, 8).astype(np.float32)
    th[8] = np.float32(th[8] * (1.0 + rng.uniform(-2e-3, 2e-3)))
    return [float(x) for x in th]


def _targets(case, tracks, seed):
    """Ring targets near the rings of the nominal geometry: centre and radius
    per (track, plane), as a reconstruction would hold them."""
    rng = np.random.default_rng([seed, 13])
    n_planes = len(_scene(case["scene"]).planes)
    tg = np.empty((tracks.n, n_planes, 4), np.float32)
    tg[..., 0:2] = rng.uniform(250.0, 480.0, (tracks.n, n_planes, 2))
    tg[..., 2] = rng.uniform(40.0, 75.0, (tracks.n, n_planes))
    tg[..., 3] = rng.random((tracks.n, n_planes)) < 0.9
    return torch.from_numpy(tg).to(DEV)


def prepare(case, seed):
    scene, kind = _scene(case["scene"]), case["kind"]
    n1, emission = _emission(case)
    ctx = rich.Context(0)
    ctx.init_geometry(scene)
    s = dict(case=case, ctx=ctx, n1=n1, emission=dict(emission, seed=seed),
             options=_trace_options(case))
    n_planes, events = len(scene.planes), case["events"]

    def outputs():
        return rich.TraceOutputs(_capacity(case) // 2, scene.pixels_per_event, n_planes, events,
                                 _capacity(case) if case.get("fate") else 0, device=DEV)

    if kind == "external":
        s["photons"] = _photon_vectors(case, seed)
        s["out"] = outputs()
        s["options"]["seed"] = seed
        return s
    tracks = _tracks(case, seed)
    s["tracks"] = rich.DeviceTracks(tracks, device=DEV)
    ctx.emit(s["tracks"], n1, **s["emission"])    # sizes the library's scratch
    if kind == "vectors":
        s["photons"] = rich.PhotonBuffers(_capacity(case), DEV)
        for v in s["photons"].t.values():
            v.zero_()
        return s
    s["out"] = outputs()
    if case.get("hits"):
        s["by_track"] = torch.zeros(s["out"].hit_capacity, 10, dtype=torch.int32, device=DEV)
    if kind == "grad":
        s["theta"] = torch.tensor(_theta(case, seed), dtype=torch.float64, requires_grad=True)
        s["targets"] = _targets(case, tracks, seed)
    elif kind == "graph":
        ctx.graph_capture(s["tracks"], s["out"], n1, **s["emission"], **s["options"])
    elif kind == "host":
        flight = case["in_flight"]
        batches = [tracks] + [_tracks(case, seed + 1000003 * k) for k in range(1, flight)]
        s["host_tracks"] = [rich.HostTracks(b) for b in batches]
        s["outs"] = [s["out"]] + [outputs() for _ in batches[1:]]
        s["host_hits"] = [torch.empty(o.hits.numel(), dtype=torch.uint8).pin_memory()
                          for o in s["outs"]]
    return s


# ---------------------------------------------------------------------- run
def _results(out):
    r = {"pixel_counts": out.pixel_counts, "event_sums": out.event_sums}
    if out.fate is not None:
        r["fate"] = out.fate
    return r


def run(s):
    case, ctx, kind = s["case"], s["ctx"], s["case"]["kind"]
    if kind == "vectors":
        ctx.emit(s["tracks"], s["n1"], photons=s["photons"], **s["emission"])
        return s["photons"].t
    if kind == "host":
        tickets = []
        for tracks, out, hits in zip(s["host_tracks"], s["outs"], s["host_hits"]):
            out.clear()
            if case["in_flight"] == 1:
                tickets.append(ctx.run_host(tracks, out, hits, s["n1"], **s["emission"],
                                            **s["options"]))
            else:
                tickets.append(ctx.run_host_async(tracks, out, hits, s["n1"], **s["emission"],
                                                  **s["options"]))
        if case["in_flight"] > 1:
            tickets = [ctx.run_wait(t) for t in tickets]
        return [dict(_results(out), n_hits=n, fates=np.array(stats["fate"]))
                for out, (n, stats) in zip(s["outs"], tickets)]
    out = s["out"]
    out.clear()
    if kind == "external":
        ctx.trace(out, photons=s["photons"], **s["options"])
        return _results(out)
    if kind == "graph":
        ctx.graph_launch()
        return _results(out)
    if kind == "grad":
        theta = s["theta"]
        theta.grad = None
        loss = rich.ring_chi2(ctx, theta, s["tracks"], s["targets"], out, sigma=1.0,
                              seed=s["emission"]["seed"])
        loss.backward()
        return {"loss": loss.detach(), "gradient": theta.grad, "pixel_counts": out.pixel_counts}
    ctx.emit(s["tracks"], s["n1"], sync=False, **s["emission"])
    ctx.trace(out, **s["options"])
    r = _results(out)
    if case.get("hits"):
        # the hit list in (track, photon) order, for fits track by track
        n, _ = ctx.hits()
        words = out.hits[: 40 * n].view(torch.int32).view(n, 10)
        order = torch.argsort(words[:, 1].long() * (1 << 32) + words[:, 2])
        hits = s["by_track"]
        torch.index_select(words, 0, order, out=hits[:n])
        r["hit_keys"] = hits[:, :5]
        r["hit_lambda"] = hits.view(torch.float32)[:, 5]
        r["hit_uv"] = hits.view(torch.float64)[:, 3:]
    return r


# --------------------------------------------------------------------- work
def _photons(case):
    k = case.get("photons")
    return case["tracks"] * (k if k else _SCENES[case["scene"]][3]) * case.get("in_flight", 1)


def work(case):
    """One pass: track records (or photon vectors) read, histograms, sums,
    fates and hits written; per photon its draws and direction (~100
    operations), per surface it meets the nearest surface, the hit and the
    response (~60 + 20 per surface of the scene tested), per detected photon
    the refined position."""
    kind = case["kind"]
    n = _photons(case)
    *_, share, met, surfaces = _SCENES[case["scene"]]
    flight = case.get("in_flight", 1)
    if kind == "vectors":
        return {"bytes": 44.0 * case["tracks"] + 40.0 * n, "flops": 100.0 * n}
    if case.get("prefilter"):
        share, met = 0.145, 0.15 * met
    scene = _scene(case["scene"])
    b = (44.0 * case["tracks"] * flight if kind != "external" else 40.0 * n)
    b += flight * case["events"] * 4.0 * scene.pixels_per_event
    b += n if case.get("fate") else 0.0
    b += 40.0 * share * n * (2.0 if case.get("hits") or kind == "host" else 1.0)
    f = n * (100.0 + met * (60.0 + 20.0 * min(surfaces, 12)))
    if case["precision"] == "refined":
        f += share * n * (3000.0 if kind == "grad" else 1000.0)
    return {"bytes": b, "flops": f}


def tolerance(case):
    """Whole numbers (counts, keys, fates) are decided in FP32: a photon
    within FP32 rounding of a mirror or pixel edge may fall on either side
    (the library's bar: at most 1e-5 of photons). Sums and positions are
    double-word where refined, FP32 where asked for; a photon that changes
    sides moves a sum by one hit."""
    kind = case["kind"]
    if kind == "vectors":
        return {"rel": 2e-7, "max": 1e-6}      # FP32 values, a few roundings each
    if kind == "grad":                         # FP32 tangents, measured 4e-8 from 64 bits
        return {"rel": 5e-7, "max": 5e-6, "differ": 1e-5}
    hits = max(1.0, _SCENES[case["scene"]][4] * _photons(case))
    rel = 1e-11 if case["precision"] == "refined" else 6e-6    # measured 2e-14 and 1.6e-6
    return {"rel": min(1e-3, rel + 2.0 / hits), "max": min(0.05, 40 * rel + 40.0 / hits),
            "differ": 2e-5}


# -------------------------------------------------------------------- exact
# The analytic scenes in plain torch, FP64: counter-based draws, emission,
# nearest surface, responses. Wavelengths and probabilities are single FP32
# operations by definition and are formed as such.
def _basis(t):
    s = torch.where(t[:, 2] >= 0, 1.0, -1.0).to(t.dtype)
    a = -1.0 / (s + t[:, 2])
    b = t[:, 0] * t[:, 1] * a
    return (torch.stack([1.0 + s * t[:, 0] ** 2 * a, s * b, -s * t[:, 0]], 1),
            torch.stack([b, s + t[:, 1] ** 2 * a, -t[:, 1]], 1))


def _philox(block, photon, track, event, seed):
    """Philox4x32-10 (Salmon et al., SC'11); 32-bit words in int64."""
    mask = 0xFFFFFFFF
    c = [torch.full_like(photon, block) if isinstance(block, int) else block, photon, track, event]
    k0, k1 = seed & mask, (seed >> 32) & mask

    def wide(m, x):                       # 32 x 32 -> (high, low), by 16-bit parts
        lo, hi = m * (x & 0xFFFF), m * (x >> 16)
        hi = hi + (lo >> 16)
        return hi >> 16, ((hi & 0xFFFF) << 16) | (lo & 0xFFFF)

    for _ in range(10):
        h0, l0 = wide(0xD2511F53, c[0])
        h1, l1 = wide(0xCD9E8D57, c[2])
        c = [h1 ^ c[1] ^ k0, l1, h0 ^ c[3] ^ k1, l0]
        k0, k1 = (k0 + 0x9E3779B9) & mask, (k1 + 0xBB67AE85) & mask
    return c


def _u24(w):
    return (w >> 8).double() / 16777216.0


def _poisson(mu, uniforms):
    """Inversion below 10, else Hoermann's PTRS (1993)."""
    if not mu > 0.0:
        return 0
    if mu < 10.0:
        u, pk, k = next(uniforms), math.exp(-mu), 0
        cdf = pk
        while cdf <= u and k < 1000:
            k += 1
            pk *= mu / k
            cdf += pk
        return k
    b = 0.931 + 2.53 * math.sqrt(mu)
    a = -0.059 + 0.02483 * b
    inv_alpha, v_r = 1.1239 + 1.1328 / (b - 3.4), 0.9277 - 3.6224 / (b - 2.0)
    for _ in range(64):
        u, v = next(uniforms) - 0.5, next(uniforms)
        us = 0.5 - abs(u)
        if not us > 0.0:
            continue
        k = math.floor((2.0 * a / us + b) * u + mu + 0.43)
        if k < 0:
            continue
        if us >= 0.07 and v <= v_r:
            return k
        if us < 0.013 and v > us:
            continue
        lhs = (math.log(v) if v > 0.0 else -math.inf) + math.log(inv_alpha) \
            - math.log(a / (us * us) + b)
        if lhs <= -mu + k * math.log(mu) - math.lgamma(k + 1.0):
            return k
    return math.floor(mu + 0.5)


def _counts(case, t, seed):
    if t.n_fixed is not None:
        return t.n_fixed.astype(np.int64)
    n1, kw = _emission(case)
    p, m = t.p.astype(np.float64), t.mass.astype(np.float64)
    if case["scene"] == "scint":
        mu = t.length.astype(np.float64) * float(np.float32(kw["yield_per_mm"]))
    else:
        nb = (1.0 + float(np.float32(n1))) * p / np.sqrt(p * p + m * m)
        band = 1e6 / kw["lambda_min"] - 1e6 / kw["lambda_max"]
        mu = t.length * 2.0 * math.pi / 137.035999 * band * np.where(
            nb > 1.0, 1.0 - 1.0 / np.maximum(nb, 1.0) ** 2, 0.0)
    blocks = 8
    ev = torch.from_numpy(t.event.astype(np.int64))
    tid = torch.from_numpy(t.id.astype(np.int64))
    words = torch.stack([w for b in range(blocks) for w in
                         _philox(b, torch.full_like(ev, 0xFFFFFFFF), tid, ev, seed)], 1)
    u = _u24(words).numpy()
    return np.array([_poisson(float(mu[i]), iter(u[i])) for i in range(t.n)], np.int64)


def _emit64(case, t, seed, n1=None):
    """Every photon of the tracks in index order, FP64."""
    counts = _counts(case, t, seed)
    total = int(counts.sum())
    track = torch.from_numpy(np.repeat(np.arange(t.n), counts)).to(DEV)
    j = torch.from_numpy(np.arange(total) - np.repeat(np.cumsum(counts) - counts, counts)).to(DEV)

    def of(a, dtype=np.float64):
        return torch.from_numpy(np.asarray(a).astype(dtype)).to(DEV)[track]

    ev, tid = of(t.event, np.int64), of(t.id, np.int64)
    w0, w1, w2, w3 = (_philox(b, j, tid, ev, seed) for b in range(4))
    d = torch.stack([of(t.dx), of(t.dy), of(t.dz)], 1)
    d = d / d.norm(dim=1, keepdim=True)
    o = torch.stack([of(t.x), of(t.y), of(t.z)], 1) + d * (_u24(w0[0]) * of(t.length))[:, None]
    phi = 2.0 * math.pi * _u24(w0[1])
    nominal, kw = _emission(case)
    f32 = np.float32
    if case["scene"] == "scint":
        tab = _scene("scint").tables[kw["spectrum_table"]]
        c = torch.from_numpy(tab["values"][: int(tab["nbins"]) + 1].copy()).to(DEV)
        u = _u24(w0[2]).float()
        k = (torch.searchsorted(c, u, right=True) - 1).clamp(0, int(tab["nbins"]) - 1)
        frac = (u - c[k]) / (c[k + 1] - c[k])
        lam = (k.float() + frac) * float(tab["p1"]) + float(tab["p0"])
        ct = 1.0 - 2.0 * _u24(w3[2])
        st = torch.sqrt((1.0 - ct * ct).clamp(min=0.0))
        dirs = torch.stack([st * torch.cos(phi), st * torch.sin(phi), ct], 1)
    else:
        inv1 = f32(1.0) / f32(kw["lambda_min"])
        span = inv1 - f32(1.0) / f32(kw["lambda_max"])
        lam = torch.ones((), device=DEV) / (float(inv1) - _u24(w0[2]).float() * float(span))
        p, m = of(t.p), of(t.mass)
        index = float(np.float32(nominal)) if n1 is None else n1
        nb = (1.0 + index) * p / torch.sqrt(p * p + m * m)
        ct = 1.0 / nb
        st = torch.sqrt(1.0 - ct * ct)
        e1, e2 = _basis(d)
        dirs = d * ct[:, None] + (e1 * torch.cos(phi)[:, None]
                                  + e2 * torch.sin(phi)[:, None]) * st[:, None]
    return dict(o=o, d=dirs, lam=lam, track=track, event=ev, track_id=tid, j=j, u_qe=_u24(w0[3]),
                u_refl=[_u24(w) for w in w1 + w2], w3=w3)


def _response(tab, lam):
    if int(tab["kind"]) == W.TABLE_CONST:
        return torch.full_like(lam, float(tab["p0"]))
    if int(tab["kind"]) == W.TABLE_GAUSS:
        x = (lam - float(tab["p1"])) / float(tab["p2"])
        return float(tab["p0"]) * torch.exp(-(x * x))
    width = torch.full((), float(tab["p1"]), device=DEV)
    b = torch.floor((lam - float(tab["p0"])) / width).long().clamp(0, int(tab["nbins"]) - 1)
    return torch.from_numpy(tab["values"].copy()).to(DEV)[b]


def _surfaces(scene, theta=None):
    """(kind, geometry, material) of every analytic surface in descriptor
    order; theta: tile tilts and radius of curvature about the fixed poles."""
    def vec(a):
        return torch.from_numpy(np.asarray(a, np.float64)).to(DEV)

    def turn(u, angle, v):
        return (v * torch.cos(angle) + torch.linalg.cross(u, v) * torch.sin(angle)
                + u * (u @ v) * (1.0 - torch.cos(angle)))

    got = []
    for i, t in enumerate(scene.spheres):
        c, a, e1, e2 = vec(t["center"]), vec(t["axis"]), vec(t["e1"]), vec(t["e2"])
        r = torch.tensor(float(t["radius"]), dtype=torch.float64, device=DEV)
        if theta is not None:
            pole, u1, u2 = c + r * a, e1, e2
            if i < 4:
                a, e1, e2 = (turn(u2, theta[2 * i + 1], turn(u1, theta[2 * i], v))
                             for v in (a, e1, e2))
            r = theta[8]
            c = pole - r * a
        edges = [[float(x) for x in e] for e in t["edges"][: int(t["n_edges"])]]
        got.append(("sphere", (c, r, a, e1, e2, float(t["cos_min"]), edges), int(t["material"])))
    for t in scene.rects:
        got.append(("rect", (vec(t["origin"]), vec(t["u_axis"]), vec(t["v_axis"]),
                             vec(t["normal"]), float(t["width"]), float(t["height"])),
                    int(t["material"])))
    return got


def _distances(surface, o, d):
    """Distances to the surface (up to two, nearest first) and their validity."""
    kind, g, _ = surface
    if kind == "rect":
        at, u, v, n, w, h = g
        t = ((at - o) @ n) / (d @ n)
        q = o + t[:, None] * d - at
        x, y = q @ u, q @ v
        return [(t, (x >= 0) & (x < w) & (y >= 0) & (y < h))]
    c, r, a, e1, e2, cos_min, edges = g
    w = o - c
    b = (w * d).sum(1)
    disc = b * b - ((w * w).sum(1) - r * r)
    sq = torch.sqrt(disc.clamp(min=0.0))
    got = []
    for t in (-b - sq, -b + sq):
        p = w + t[:, None] * d
        ok = (disc >= 0) & (p @ a / r >= cos_min)
        x, y = p @ e1, p @ e2
        for ea, eb, ec in edges:
            ok = ok & (ea * x + eb * y <= ec)
        got.append((t, ok))
    return got


def _normal(surface, p):
    return (surface[1][0] - p) / surface[1][1] if surface[0] == "sphere" \
        else surface[1][3].expand_as(p)


def _trace64(scene, ph, surfaces):
    """Nearest-surface propagation of all photons: the detected ones' indices,
    planes, plane coordinates and sequences of mirrors met, and all fates."""
    n = len(ph["lam"])
    o, d = ph["o"].clone(), ph["d"].clone()
    fate = torch.zeros(n, dtype=torch.uint8, device=DEV)
    skip = torch.full((n,), -1, device=DEV)
    turns = torch.zeros(n, dtype=torch.long, device=DEV)
    path = torch.full((n, 8), -1, device=DEV)
    plane = torch.full((n,), -1, device=DEV)
    uv = torch.zeros(n, 2, dtype=torch.float64, device=DEV)
    refl = torch.stack(ph["u_refl"], 1)
    for step in range(16):
        live = torch.nonzero(fate == 0).squeeze(1)
        if not len(live):
            break
        lo, ld = o[live], d[live]
        best = torch.full((len(live),), math.inf, dtype=torch.float64, device=DEV)
        prim = torch.full((len(live),), -1, device=DEV)
        for k, s in enumerate(surfaces):
            for t, ok in _distances(s, lo, ld):
                ok = ok & (t > 1e-3) & (t < best) & (skip[live] != k)
                best = torch.where(ok, t, best)
                prim = torch.where(ok, k, prim)
        fate[live[prim < 0]] = 1
        for k, s in enumerate(surfaces):
            at = torch.nonzero(prim == k).squeeze(1)
            if not len(at):
                continue
            i = live[at]
            p = lo[at] + best[at][:, None] * ld[at]
            nrm = _normal(s, p)
            dn = (ld[at] * nrm).sum(1)
            front = dn < 0
            m = scene.materials[s[2]]
            kind = int(m["kind"])
            go = torch.ones_like(front)
            if kind == W.MAT_ABSORBER:
                fate[i], go = 3, torch.zeros_like(front)
            else:
                pr = _response(scene.tables[int(m["table"])], ph["lam"][i]).double()
            if kind == W.MAT_MIRROR:
                full = turns[i] >= 8
                ok = refl[i, turns[i].clamp(max=7)] < pr
                fate[i] = torch.where(~front, 3, torch.where(full, 6, torch.where(ok, 0, 2))).to(
                    torch.uint8)
                go = front & ~full & ok
                r = ld[at] - 2.0 * dn[:, None] * nrm
                d[i[go]] = (r / r.norm(dim=1, keepdim=True))[go]
                path[i[go], turns[i[go]]] = k
                turns[i[go]] += 1
            elif kind == W.MAT_DETECTOR:
                ok = ph["u_qe"][i] < pr
                fate[i] = torch.where(~front, 0, torch.where(ok, 5, 4)).to(torch.uint8)
                go = ~front
                q = p - s[1][0]
                plane[i] = int(m["plane"])
                uv[i] = torch.stack([q @ s[1][1], q @ s[1][2]], 1)
            o[i[go]] = p[go]
            skip[i[go]] = k
        still = live[fate[live] == 0]
        if step == 15:
            fate[still] = 7
    hit = torch.nonzero(fate == 5).squeeze(1)
    return dict(hit=hit, plane=plane[hit], uv=uv[hit], path=path[hit], fate=fate)


def _exact_gradient(case, seed):
    scene, t = _scene(case["scene"]), _tracks(case, seed)
    theta = torch.tensor(_theta(case, seed), dtype=torch.float64, device=DEV, requires_grad=True)
    ph = _emit64(case, t, seed, n1=theta[9])
    surfaces = _surfaces(scene, theta)
    with torch.no_grad():
        still = {k: v.detach() if torch.is_tensor(v) else v for k, v in ph.items()}
        det = _trace64(scene, still, surfaces)
    i = det["hit"]
    o, d = ph["o"][i], ph["d"][i]
    for k in range(8):
        for q in torch.unique(det["path"][:, k]).tolist():
            if q < 0:
                continue
            at = torch.nonzero(det["path"][:, k] == q).squeeze(1)
            t_hit = _distances(surfaces[q], o[at], d[at])[-1][0]    # the concave side's exit root
            p = o[at] + t_hit[:, None] * d[at]
            nrm = _normal(surfaces[q], p)
            r = d[at] - 2.0 * (d[at] * nrm).sum(1)[:, None] * nrm
            o, d = o.index_copy(0, at, p), d.index_copy(0, at, r / r.norm(dim=1, keepdim=True))
    uv = torch.zeros(len(i), 2, dtype=torch.float64, device=DEV)
    for s in surfaces:
        if int(scene.materials[s[2]]["kind"]) != W.MAT_DETECTOR:
            continue
        at = torch.nonzero(det["plane"] == int(scene.materials[s[2]]["plane"])).squeeze(1)
        q = o[at] + _distances(s, o[at], d[at])[0][0][:, None] * d[at] - s[1][0]
        uv = uv.index_copy(0, at, torch.stack([q @ s[1][1], q @ s[1][2]], 1))
    w3 = [w[i] for w in ph["w3"]]
    rad = torch.sqrt(-2.0 * torch.log(((w3[0] >> 8).double() + 0.5) / 16777216.0))
    ang = 2.0 * math.pi * _u24(w3[1])
    h = uv + torch.stack([rad * torch.cos(ang), rad * torch.sin(ang)], 1)
    tg = _targets(case, t, seed).double()[ph["track"][i], det["plane"]]
    rho = (h - tg[:, :2]).norm(dim=1) - tg[:, 2]
    loss = (rho * rho)[tg[:, 3] > 0].mean()
    loss.backward()
    return {"loss": loss.detach(), "gradient": theta.grad, "pixel_counts": None}


def exact(case, seed):
    if case["kind"] == "vectors":
        ph = _emit64(case, _tracks(case, seed), seed)
        r = {k: ph["o"][:, i] for i, k in enumerate("xyz")}
        r.update({"d" + k: ph["d"][:, i] for i, k in enumerate("xyz")}, lambda_=ph["lam"].double())
        pad = _capacity(case) - len(ph["lam"])
        r = {k: torch.nn.functional.pad(v, (0, pad)) for k, v in r.items()}
        return dict(r, event=None, track=None, photon=None)
    if case["kind"] == "grad":
        return _exact_gradient(case, seed)
    scene = _scene(case["scene"])
    if case["kind"] != "step" or scene.n_triangles or case.get("prefilter") \
            or case.get("dispersive"):
        return None                              # meshes and wavelength-dependent angles
    ph = _emit64(case, _tracks(case, seed), seed)
    det = _trace64(scene, ph, _surfaces(scene))
    i, n_planes = det["hit"], len(scene.planes)
    sums = torch.zeros(case["events"] * n_planes, 4, dtype=torch.float64, device=DEV)
    rows = torch.stack([torch.ones(len(i), dtype=torch.float64, device=DEV), det["uv"][:, 0],
                        det["uv"][:, 1], ph["lam"][i].double()], 1)
    sums.index_add_(0, ph["event"][i] * n_planes + det["plane"], rows)
    return {"pixel_counts": None, "event_sums": sums.reshape(-1),
            "fate": None}
