"""The work that programs have this library do, as cases to be measured: sizes, inputs, one pass
through the public entry points, the work it cannot do without, and its results in 64 bits.

A case names an entry point (`call`), a detector, the number of events and of tracks per event and
the search's options.  Inputs are synthetic events of `synth`; a batch of many events is put
together on the GPU from a smaller simulated sample, copied under rotations about the beam axis
and reflections (the cylinders, the disks and the field are the same under both), so that making
it takes less than a second at every size.
"""
import math

import numpy as np
import torch

from paper_2312_11728_gb300 import mkgb, pipeline, synth as S
from paper_2312_11728_gb300.fitgrad import FitChi2

SAMPLE = 4000          # tracks simulated for a batch of cylinders and disks, at most
MIN_HITS = 7           # of a track that is seeded, fitted and counted
MAX_CASE_TRACKS = 1_280_000

# The options of every case: the search's own defaults otherwise (6 candidates per seed).
_BASE = dict(detector="phase2", events=1, tracks=20000, uneven=False, cands=6)


def _case(name, call, **kw):
    return dict(_BASE, call=call, name=name, **kw)


def listed():
    return [
        # one small event in one call, as a trigger or a test beam would ask for it: launches and latency
        _case("run_barrel_1k", "run", detector="barrel", tracks=1000),
        # one full event, processed as soon as it is read
        _case("run_phase2_1ev", "run"),
        # the throughput batch of offline reconstruction: hits in, seeds, search, final fit
        _case("run_phase2_64ev", "run", events=64),
        # events of uneven size, as a fill delivers them, in one call
        _case("run_uneven_256ev", "run", events=256, tracks=8000, uneven=True),
        # a fast iteration that keeps two candidates per seed instead of six
        _case("run_two_cands_16ev", "run", events=16, cands=2),
        # a tracker with tilted and planar modules: hits on their planes, overlap hits picked up
        _case("run_modular_2ev", "modular", detector="modular", events=2, tracks=6000),
        # host arrays in, host arrays out: the call of a program that keeps its events in host memory
        _case("run_host_16ev", "host", events=16),
        # hit preparation and seed states handed back, for a program with its own track finding
        _case("seed_32ev", "seed", events=32),
        # the final fit of tracks found elsewhere, a tenth of them curling
        _case("fit_loopers_1m", "fit", detector="loopers", events=50),
        # refit backwards and look for the inner hits that seeding further out left behind
        _case("backward_16ev", "backward", events=16),
        # one step of alignment: the chi2 and its derivative in every alignment and thickness parameter
        _case("align_100k", "grad", detector="endcap", events=5),
        # duplicates among seeds and among found tracks
        _case("cleaning_32ev", "clean", events=32),
    ]


def draw(rng):
    call = rng.choice(["run", "run", "run", "modular", "host", "seed", "fit", "backward", "grad", "clean"])
    most = {"modular": 12000, "grad": 100_000, "host": 320_000, "backward": 320_000, "seed": 640_000,
            "clean": 640_000}.get(call, MAX_CASE_TRACKS)
    total = math.exp(rng.uniform(math.log(500), math.log(most)))
    per_event = math.exp(rng.uniform(math.log(300), math.log(min(25000, total) if total > 400 else 400)))
    if call == "modular":
        per_event = max(per_event, total / 2)
    per_event = max(per_event, total / 256)
    c = dict(_BASE, call=call, events=max(1, int(total / per_event)), tracks=int(per_event) | 1)
    if call == "run":
        c["detector"] = rng.choice(["phase2", "phase2", "barrel"])
        c["uneven"] = rng.random() < 0.5
        c["cands"] = rng.choice([1, 2, 4, 6, 6])
    elif call in ("modular", "fit", "grad"):
        c["detector"] = {"modular": "modular", "fit": rng.choice(["loopers", "phase2"]), "grad": "endcap"}[call]
    return c


# ------------------------------------------------------------------------------------------ inputs

def _geometry(detector):
    if detector == "barrel":
        return S.geometry_barrel()
    if detector == "modular":
        return S.geometry_phase2_modular_disks()
    return S.geometry_phase2()


def _sample(detector, geom, n, seed, event=0):
    """One simulated event of n tracks; the noise hits in proportion (50,000 per 20,000 tracks on
    the cylinders and disks, 200 per layer and 1,000 tracks in the barrel alone)."""
    if detector == "barrel":
        return S.simulate_event(geom, n, seed, event, eta_max=1.0, noise_per_layer=max(1, n // 5))
    kw = dict(pt_sampler=S.sample_pt_phase2, eta_max=3.0, noise_total=int(2.5 * n))
    if detector == "loopers":
        kw.update(pt_sampler=S.sample_pt_loopers, noise_total=0)
    if detector == "endcap":
        kw.update(eta_min=0.0, noise_total=0)
    return S.simulate_event(geom, n, seed, event, **kw)


def _counts(case):
    """Tracks per event: the case's own, whatever the seed."""
    n, e = case["tracks"], case["events"]
    if not case["uneven"]:
        return np.full(e, n)
    return np.clip(np.random.default_rng([n, e]).poisson(n, e), 200, 25000)


def _more(n):
    """Tracks to simulate so that n of them have MIN_HITS (almost all have)."""
    return int(1.03 * n) + 16


def _first(n_hits, n):
    """The first n tracks with MIN_HITS."""
    t = np.nonzero(n_hits >= MIN_HITS)[0][:n]
    if len(t) < n:
        raise RuntimeError(f"{len(t)} of {n} tracks have {MIN_HITS} hits")
    return t


def _dev(a, dtype=None):
    t = torch.from_numpy(np.ascontiguousarray(a)).cuda()
    return t if dtype is None else t.to(dtype)


def _rotate(xyz, cov, ang, mirror):
    """Points and packed covariances (xx, yx, yy, zx, zy, zz) turned about z by ang after y -> mirror y."""
    c, s = torch.cos(ang), torch.sin(ang)
    x, y, z = xyz[:, 0], mirror * xyz[:, 1], xyz[:, 2]
    a, b, d, e, f, g = (cov[:, k] for k in range(6))
    b, f = mirror * b, mirror * f
    out = torch.stack([c * x - s * y, s * x + c * y, z], 1)
    v = torch.stack([c * c * a - 2 * c * s * b + s * s * d, c * s * a + (c * c - s * s) * b - c * s * d,
                     s * s * a + 2 * c * s * b + c * c * d, c * e - s * f, s * e + c * f, g], 1)
    return out, v


def _batch(case, geom, seed, align=None):
    """A batch on the GPU: hits grouped by (event, layer), seed hits, and every track's known
    assignment with a starting state (the inputs of mkgb_run)."""
    rng = np.random.default_rng([seed, 1])
    counts = _counts(case)
    L = geom.n_layers
    nb = int(min(counts.max(), 20000 if case["call"] == "fit" else SAMPLE))
    ev = _sample(case["detector"], geom, _more(nb), seed)
    fl, fh, fp0, fc0, _, nh, sel = S.fit_workload(ev, seed=seed)
    use = _first(nh, nb)
    fl, fh, fp0, fc0 = fl[use], fh[use], fp0[use], fc0[use]
    number = np.full(len(ev.track_q), -1)      # of each simulated track among the ones used
    number[sel[use]] = np.arange(nb)
    hit_track = np.where(ev.hit_track >= 0, number[ev.hit_track], -1)
    # copies of the sample: (event, tracks taken), then its rotation and reflection
    ov_event, ov_n = [], []
    for e, n in enumerate(counts):
        k = -(-int(n) // nb)
        for j in range(k):
            ov_event.append(e)
            ov_n.append(int(n) * (j + 1) // k - int(n) * j // k)
    O = len(ov_event)
    ov_event, ov_n = _dev(np.array(ov_event)), _dev(np.array(ov_n))
    ang = _dev(rng.uniform(-np.pi, np.pi, O))
    mir = _dev(np.where(rng.random(O) < 0.5, -1.0, 1.0))
    gen = torch.Generator("cuda").manual_seed(seed)
    rank = torch.rand((O, nb), generator=gen, device="cuda").argsort(1).argsort(1)
    taken = rank < ov_n[:, None]                                                  # [O, tracks]
    ht = _dev(hit_track)
    noise = torch.rand((O, ht.numel()), generator=gen, device="cuda") < (ov_n / nb)[:, None]
    keep = torch.where(ht >= 0, taken[:, ht.clamp(min=0)], noise)
    lay = torch.bucketize(torch.arange(ht.numel(), device="cuda"), _dev(ev.layer_off[1:]), right=True)
    o, h = keep.nonzero(as_tuple=True)
    seg = ov_event[o] * L + lay[h]
    order = seg.argsort(stable=True)
    o, h, seg = o[order], h[order], seg[order]
    xyz, cov = _rotate(_dev(ev.hit_xyz, torch.float64)[h], _dev(ev.hit_cov, torch.float64)[h], ang[o], mir[o])
    if align is not None:
        al = align[lay[h]]
        c = torch.zeros_like(xyz)
        c[:, 2] = (_dev(geom.pos) * _dev(geom.kind))[lay[h]]   # kind 1: a disk, turned about its own centre
        xyz = xyz + al[:, :3] + torch.linalg.cross(al[:, 3:], xyz - c)
    where = torch.full((O, ht.numel()), -1, dtype=torch.int64, device="cuda")
    where[o, h] = torch.arange(h.numel(), device="cuda")
    seg_off = torch.zeros(len(counts) * L + 1, dtype=torch.int64, device="cuda")
    seg_off[1:] = torch.bincount(seg, minlength=len(counts) * L).cumsum(0)

    oo, r = taken.nonzero(as_tuple=True)
    loc = _dev(fh).long()[r]
    hits = torch.where(loc >= 0, where[oo[:, None], loc.clamp(min=0)], -1).int().contiguous()
    p0, m = _dev(fp0, torch.float64)[r], mir[oo]
    xy, _ = _rotate(p0[:, :3], torch.zeros((len(r), 6), dtype=torch.float64, device="cuda"), ang[oo], m)
    phi = torch.remainder(m * p0[:, 4] + ang[oo] + math.pi, 2 * math.pi) - math.pi
    p0 = torch.stack([xy[:, 0], xy[:, 1], xy[:, 2], m * p0[:, 3], phi, p0[:, 5]], 1)
    return dict(n_events=len(counts), seg_off=seg_off.cpu().numpy(), xyz=xyz.float().contiguous(),
                cov=cov.float().contiguous(), seeds=hits[:, :3].contiguous(), layers=_dev(fl)[r].int().contiguous(), hits=hits,
                p0=p0.float().contiguous(), c0=_dev(fc0, torch.float32)[r].contiguous(), event=ov_event[oo].int())


def _modular_batch(case, geom, seed):
    """Events of the modular tracker, simulated one by one (its modules are no rotation of themselves)."""
    n = case["tracks"]
    evs = [_sample("modular", geom, _more(n), seed, e) for e in range(case["events"])]
    b = S.concat_events(evs, geom.n_layers)
    fi = pipeline.fit_inputs(b, seed)
    t = np.concatenate([np.nonzero(fi.event == e)[0][_first((fi.layers[fi.event == e] >= 0).sum(1), n)]
                        for e in range(case["events"])])
    return dict(n_events=b.n_events, seg_off=b.hit_off, xyz=_dev(b.hit_xyz), cov=_dev(b.hit_cov),
                seeds=_dev(fi.hits[t, :3]), layers=_dev(fi.layers[t]), hits=_dev(fi.hits[t]), p0=_dev(fi.p0[t]),
                c0=_dev(fi.c0[t]), hit_module=_dev(b.hit_mod))


def _fit_out(n, device="cuda", pin=False):
    z = lambda *s, t=torch.float32: torch.zeros(s, dtype=t, device=device, pin_memory=pin)
    return dict(p=z(n, 6), c=z(n, 21), chi2=z(n), status=z(n, t=torch.int32))


def _tracks_out(n, width, pin=False, ovl=False):
    if not pin:
        return mkgb.alloc_tracks(n, width, "cuda", ovl=ovl)
    t = mkgb.alloc_tracks(n, width)
    return {k: torch.from_numpy(v).pin_memory() for k, v in t.items()}


def _make(case, seed):
    """The geometry and the batch of a case (and the starting alignment of its derivative)."""
    geom = _geometry(case["detector"])
    if case["call"] == "modular":
        return geom, _modular_batch(case, geom, seed)
    if case["call"] != "grad":
        return geom, _batch(case, geom, seed)
    rng = np.random.default_rng([seed, 2])
    L = geom.n_layers
    true = np.concatenate([rng.normal(0, 50e-4, (L, 3)), rng.normal(0, 1e-4, (L, 3))], 1)
    b = _batch(case, geom, seed, align=_dev(true))
    # the alignment a program has reached so far: half of the true one, thicknesses off by up to 20%
    b["align"] = _dev(-0.5 * true, torch.float32)
    b["xscale"] = _dev(rng.uniform(0.8, 1.2, L), torch.float32)
    return geom, b


def prepare(case, seed):
    geom, b = _make(case, seed)
    s = dict(b, case=case, geom=geom, call=case["call"])
    s["ctx"] = pipeline.make_context(geom, S.default_params(max_cands=case["cands"]))
    n, t, width = int(b["seeds"].shape[0]), int(b["layers"].shape[0]), geom.max_plan
    call = case["call"]
    if call == "host":
        for k in ("xyz", "cov", "seeds", "layers", "hits", "p0", "c0"):
            s[k] = b[k].cpu().pin_memory()
        s["out"], s["fit"] = _tracks_out(n, width, pin=True), _fit_out(t, "cpu", pin=True)
    elif call in ("run", "modular"):
        s["out"], s["fit"] = _tracks_out(n, width, ovl=call == "modular"), _fit_out(t)
    elif call == "seed":
        z = lambda w, d: torch.zeros((n, w), dtype=d, device="cuda")
        s["state"], s["state_cov"], s["info"] = z(6, torch.float32), z(21, torch.float32), z(3, torch.int32)
    else:
        # hits loaded once, as by a program that fits or cleans the tracks of one batch
        s["ctx"].load_hits(b["n_events"], b["seg_off"], b["xyz"], b["cov"])
        if call == "fit":
            s["fit"] = _fit_out(t)
        elif call == "backward":
            s["layers"], s["hits"] = _outer(b["layers"]), _outer(b["hits"])
            s["first"] = s["layers"][:, 0].contiguous()
            s["fit"], s["back"], s["out"] = _fit_out(t), _fit_out(t), _tracks_out(t, width)
        elif call == "grad":
            s["leaves"] = [s[k].clone().requires_grad_() for k in ("align", "xscale", "p0")]
        elif call == "clean":
            _duplicates(s, seed)
    return s


def _outer(rows):
    """Layer or hit lists without their first three entries."""
    return torch.cat([rows[:, 3:], torch.full_like(rows[:, :3], -1)], 1).contiguous()


def _duplicates(s, seed):
    """Two seeds per track (its 1st, 2nd, 3rd and its 1st, 2nd, 4th hits) and two found tracks: one
    with all its hits, one that lost up to half of them to hits of the next track."""
    g = torch.Generator("cuda").manual_seed(seed)
    H = s["hits"]
    s["seeds"] = torch.cat([H[:, :3], H[:, [0, 1, 3]]]).contiguous()
    other = torch.roll(H, -1, 0)
    lost = torch.rand(H.shape, generator=g, device="cuda") < 0.5 * torch.rand((len(H), 1), generator=g, device="cuda")
    s["rows"] = torch.cat([H, torch.where(lost & (H >= 0), other, H)]).contiguous()
    s["score"] = torch.rand(len(s["rows"]), generator=g, device="cuda") * 60
    z = lambda n: torch.zeros(n, dtype=torch.int32, device="cuda")
    s["keep_seeds"], s["keep_rows"] = z(len(s["seeds"])), z(len(s["rows"]))


# ------------------------------------------------------------------------------------------ one pass

def run(s):
    ctx, call = s["ctx"], s["call"]
    if call in ("run", "modular", "host"):
        f = s["fit"]
        more = {"hit_module": s["hit_module"]} if call == "modular" else {}
        (ctx.run_host if call == "host" else ctx.run)(
            s["n_events"], s["seg_off"], s["xyz"], s["cov"], s["seeds"], s["out"], s["layers"], s["hits"], s["p0"],
            s["c0"], f["p"], f["c"], f["chi2"], f["status"], **more)
        return {"tracks": s["out"], "fit": f}
    if call == "seed":
        ctx.load_hits(s["n_events"], s["seg_off"], s["xyz"], s["cov"])
        ctx.seed(s["seeds"], s["state"], s["state_cov"], s["info"])
        return {"state": s["state"], "cov": s["state_cov"], "info": s["info"]}
    if call == "grad":
        align, xscale, p0 = s["leaves"]
        for t in s["leaves"]:
            t.grad = None
        total, status = FitChi2.apply(align, xscale, p0, ctx, s["layers"], s["hits"], s["c0"])
        total.backward()
        return {"chi2": total.detach(), "align": align.grad, "xscale": xscale.grad, "p0": p0.grad, "status": status}
    if call == "clean":
        ctx.clean_seeds(s["seeds"], s["keep_seeds"])
        ctx.remove_duplicates(s["rows"], s["score"], s["keep_rows"], min_hits=6, frac=0.5)
        return {"seeds": s["keep_seeds"], "tracks": s["keep_rows"]}
    f = s["fit"]
    ctx.fit(s["layers"], s["hits"], s["p0"], s["c0"], f["p"], f["c"], f["chi2"], f["status"])
    if call == "fit":
        return {"fit": f}
    b = s["back"]
    ctx.fit_backward(s["layers"], s["hits"], f["p"], f["c"], b["p"], b["c"], b["chi2"], b["status"])
    ctx.build_backward(s["event"], s["first"], b["p"], b["c"], s["out"])
    return {"fit": f, "back": b, "tracks": s["out"]}


# ------------------------------------------------------------------------------------------ the work

def work(case):
    """Bytes: inputs and outputs of the pass, each once.  Flops: per track the sizes that the events
    have on average (hits, searched layers), and per Kalman step the multiply-adds of its formulas:
    the transport of a 6 x 6 covariance to a surface (~400), the helix step with its Jacobian and
    material (~300), chi2 (~100) and update (~350 in Joseph form)."""
    t = case["events"] * case["tracks"]
    barrel = case["detector"] == "barrel"
    hits_tr = 10 if barrel else 12.4          # hits of a track
    hits = t * (hits_tr + (0 if case["detector"] in ("loopers", "endcap") else 2.0 if barrel else 2.5))
    width = 10 if barrel else 22
    step, upd = 1600, 700
    fit = t * (hits_tr * 8 + 108 + 116)       # its hit and layer lists, state in, state out
    fit_fl = t * hits_tr * (step + upd)
    seed = t * 12
    seed_fl = t * 3 * (step + upd)
    tracks = t * (6 + 21 + 4 + width) * 4
    # candidates that live on average at each of the layers after the seed's
    search_fl = t * (hits_tr - 3) * (step + upd) * (1 + 0.5 * (case["cands"] - 1))
    call = case["call"]
    if call in ("run", "modular", "host"):
        return {"bytes": hits * 36 + seed + tracks + fit, "flops": fit_fl + seed_fl + search_fl}
    if call == "seed":
        return {"bytes": hits * 36 + seed + t * 120, "flops": seed_fl}
    if call == "fit":
        return {"bytes": t * hits_tr * 36 + fit, "flops": fit_fl}
    if call == "backward":
        return {"bytes": t * 9 * 36 + 3 * fit + tracks, "flops": 2 * fit_fl + t * 3 * (step + upd)}
    if call == "grad":
        # a derivative by reverse mode costs a small multiple of the value
        return {"bytes": t * hits_tr * 36 + fit + t * 24, "flops": 5 * fit_fl}
    return {"bytes": t * (6 + 4 * hits_tr + 4) * 4 + t * 4, "flops": 10.0 * t}


# ------------------------------------------------------------------------------------------ 64 bits
#
# The fits, the seed states and the derivative written out in FP64 with torch, from the formulas:
# every crossing is solved in closed form (circle and circle, line and plane), the covariance is
# kept in the global frame, the update is the Joseph form.  The search has no such value here: its
# outputs hang on the order of its candidates.

C_LIGHT, M_PI, M_E = 0.00299792458, 0.13957039, 0.51099895e-3
DET_K, DET_ZA, DET_RHO, DET_X0, DET_I = 0.307075, 0.49848, 2.329, 9.37, 173.0e-9


def _tri(c):
    """Packed lower triangle [n, m(m+1)/2] -> symmetric [n, m, m]."""
    m = {21: 6, 6: 3}[c.shape[1]]
    at = torch.tensor([[max(i, j) * (max(i, j) + 1) // 2 + min(i, j) for j in range(m)] for i in range(m)],
                      device=c.device)
    return c[:, at]


def _pack(C):
    i, j = torch.tril_indices(6, 6, device=C.device)
    return C[:, i, j]


def _turn(x, y, phi, om, far):
    """The turn from phi to the circle's point of largest (far) or smallest radius, in [0, 2 pi)."""
    cx, cy, sg = x - torch.sin(phi) / om, y + torch.cos(phi) / om, torch.sign(om)
    return torch.remainder((torch.atan2(sg * cx, -sg * cy) + (0 if far else math.pi) - phi) * sg, 2 * math.pi)


def _cross(p, disk, pos, lo, hi, om, back):
    """Path length (signed) to the layer and whether it is crossed; no derivative."""
    x, y, z, _, phi, th = p.unbind(1)
    # cylinders: the intersection of two circles
    cx, cy, rho = x - torch.sin(phi) / om, y + torch.cos(phi) / om, 1 / om.abs()
    d = torch.hypot(cx, cy)
    a = (rho * rho - pos * pos + d * d) / (2 * d)
    h = torch.sqrt((rho * rho - a * a).clamp(min=0))
    ex, ey = -cx / d, -cy / d
    s = torch.full_like(x, math.inf)
    way = -1.0 if back else 1.0
    for sign in (1.0, -1.0):
        px, py = a * ex - sign * h * ey, a * ey + sign * h * ex
        psi = torch.atan2(om * px, -om * py)
        t = torch.remainder((psi - phi) * torch.sign(om) * way, 2 * math.pi) * rho
        s = torch.minimum(s, torch.where(t > 1e-9, t, math.inf))
    gap = pos * pos - x * x - y * y
    out = x * torch.cos(phi) + y * torch.sin(phi) > 0
    okc = ((d - rho).abs() <= pos) & (pos <= d + rho) & ((gap < 0) & out if back else gap > 0) & torch.isfinite(s)
    if back:
        okc &= s <= torch.remainder(-_turn(x, y, phi, om, False) * 1.0, 2 * math.pi) * rho
    else:
        okc &= s <= _turn(x, y, phi, om, True) * rho
    s = way * torch.where(torch.isfinite(s), s, 0.0)
    for _ in range(3):   # the root to the last bits
        dx, dy = _chord(phi, om, s)
        g = 2 * (x * dx + y * dy) + dx * dx + dy * dy - gap
        dg = 2 * ((x + dx) * torch.cos(phi + om * s) + (y + dy) * torch.sin(phi + om * s))
        s = s - torch.where(okc & (dg.abs() > 1e-9), g / dg, 0.0)
    # disks: the plane
    sd = (pos - z) * torch.tan(th)
    turn = torch.remainder(-_turn(x, y, phi, om, False), 2 * math.pi) if back else _turn(x, y, phi, om, True)
    okd = (sd * way > 0) & (sd.abs() <= turn * rho)
    s, ok = torch.where(disk, sd, s), torch.where(disk, okd, okc)
    s = torch.where(ok, s, 0.0)
    dx, dy = _chord(phi, om, s)
    xn, yn, zn = x + dx, y + dy, z + s / torch.tan(th)
    v = torch.where(disk, torch.hypot(xn, yn), zn)
    outward = xn * torch.cos(phi + om * s) + yn * torch.sin(phi + om * s) >= 0
    return s, ok & (v >= lo) & (v <= hi) & (outward | ~disk)


def _chord(phi, om, s):
    h = 0.5 * om * s
    c = s * torch.sinc(h / math.pi)
    return c * torch.cos(phi + h), c * torch.sin(phi + h)


def _step(p, C, lay, bz, on, back=False, xscale=None):
    """States p [n, 6] and covariances C moved to the layers lay (kind, pos, lo, hi, x/X0 per track)
    where `on`; returns the new ones and whether the layer was crossed (2: stopped in it)."""
    kind, pos, lo, hi, xx0 = lay
    disk = kind == 1
    cB = C_LIGHT * bz
    om = -cB * p[:, 3]
    with torch.no_grad():
        s, ok = _cross(p, disk, pos, lo, hi, om, back)
        ok &= on
        s = torch.where(ok, s, 0.0)
    x, y, z, k, phi, th = p.unbind(1)
    # one Newton step from the root: the value stays, the derivative is the implicit function's
    dx, dy = _chord(phi, om, s)
    sp, cp, cot = torch.sin(phi + om * s), torch.cos(phi + om * s), 1 / torch.tan(th)
    g = torch.where(disk, z + s * cot - pos, ((x + dx) ** 2 + (y + dy) ** 2 - pos * pos))
    dg = torch.where(disk, cot, 2 * ((x + dx) * cp + (y + dy) * sp)).detach()
    s = s - torch.where(ok, g / torch.where(dg == 0, 1.0, dg), 0.0)
    a = om * s
    dx, dy = _chord(phi, om, s)
    sp, cp = torch.sin(phi + a), torch.cos(phi + a)
    st, ct = torch.sin(th), torch.cos(th)
    xn, yn, zn = x + dx, y + dy, z + s * cot
    # Jacobian: fixed path length, then the path length's own change
    h = 0.5 * a
    sinc = torch.sinc(h / math.pi)
    small = h.abs() < 0.05
    hs = torch.where(small, 1.0, h)
    dsinc = torch.where(small, h * (-1 / 3 + h * h * (1 / 30 - h * h / 840)), (torch.cos(h) - sinc) / hs)
    ch, sh = torch.cos(phi + h), torch.sin(phi + h)
    n = len(p)
    one, zero = torch.ones(n, dtype=p.dtype, device=p.device), torch.zeros(n, dtype=p.dtype, device=p.device)
    A03 = -cB * s * s * 0.5 * (dsinc * ch - sinc * sh)
    A13 = -cB * s * s * 0.5 * (dsinc * sh + sinc * ch)
    A25 = -s / (st * st)
    rows = [torch.stack([one, zero, zero, A03, -dy, zero], 1), torch.stack([zero, one, zero, A13, dx, zero], 1),
            torch.stack([zero, zero, one, zero, zero, A25], 1)]
    r = torch.hypot(xn, yn)
    nrm = torch.stack([torch.where(disk, 0.0, xn / r), torch.where(disk, 0.0, yn / r), torch.where(disk, 1.0, 0.0)], 1)
    nA = sum(nrm[:, q, None] * rows[q] for q in range(3))
    nf = nrm[:, 0] * cp + nrm[:, 1] * sp + nrm[:, 2] * cot
    ds = -nA / torch.where(nf == 0, 1.0, nf)[:, None]
    J = torch.stack([rows[0] + cp[:, None] * ds, rows[1] + sp[:, None] * ds, rows[2] + cot[:, None] * ds,
                     torch.stack([zero, zero, zero, one, zero, zero], 1),
                     torch.stack([zero, zero, zero, -cB * s, one, zero], 1) + om[:, None] * ds,
                     torch.stack([zero, zero, zero, zero, zero, one], 1)], 1)
    Cn = J @ C @ J.transpose(1, 2)
    # material
    inc = torch.where(disk, ct.abs(), ((xn * cp + yn * sp) * st / r).abs())
    tt = xx0 * torch.clamp(1 / inc.clamp(min=1e-9), max=10.0)
    if xscale is not None:
        tt = tt * xscale
    mat = tt.detach() > 0
    ts = torch.where(mat, tt, 1.0)
    pm = 1 / (k.abs() * st)
    e2 = pm * pm + M_PI * M_PI
    b2, e = pm * pm / e2, torch.sqrt(e2)
    th0 = 0.0136 / (torch.sqrt(b2) * pm) * torch.sqrt(ts) * (1 + 0.038 * torch.log(ts / b2))
    bg2, gam, rme = pm * pm / M_PI ** 2, e / M_PI, M_E / M_PI
    tmax = 2 * M_E * bg2 / (1 + 2 * gam * rme + rme * rme)
    de = DET_K * DET_ZA / b2 * (0.5 * torch.log(2 * M_E * bg2 * tmax / DET_I ** 2) - b2) * DET_RHO * ts * DET_X0 * 1e-3
    en = e + de if back else e - de
    stopped = mat & (en <= M_PI)
    en = torch.where(en > M_PI * 1.0000001, en, 2 * M_PI)
    f = torch.where(mat, pm / torch.sqrt((en - M_PI) * (en + M_PI)), 1.0)
    t2, kc = torch.where(mat, th0 * th0, 0.0), k * cot
    Q = torch.zeros_like(Cn)
    Q[:, 4, 4], Q[:, 5, 5], Q[:, 3, 3] = t2 / (st * st), t2, kc * kc * t2
    Q[:, 3, 5] = Q[:, 5, 3] = -kc * t2
    sc = torch.ones((n, 6), dtype=p.dtype, device=p.device)
    sc[:, 3] = f
    Cn = (Cn + Q) * sc[:, :, None] * sc[:, None, :]
    pn = torch.stack([xn, yn, zn, k * f, torch.remainder(phi + a + math.pi, 2 * math.pi) - math.pi, th], 1)
    good = ok & ~stopped
    return (torch.where(good[:, None], pn, p), torch.where(good[:, None, None], Cn, C),
            torch.where(ok, torch.where(stopped, 2, 1), 0))


def _update(p, C, m, V, on, dm=None):
    """Joseph-form update with hits (m, V) where `on`: state, covariance, chi2 (0 elsewhere)."""
    eye = torch.eye(6, dtype=p.dtype, device=p.device)
    Sm = torch.where(on[:, None, None], C[:, :3, :3] + V, eye[:3, :3])
    r = m - p[:, :3]
    if dm is not None:
        r = r + dm
    W = torch.linalg.inv(Sm)
    x2 = torch.where(on, (r[:, None, :] @ W @ r[:, :, None])[:, 0, 0], 0.0)
    K = C[:, :, :3] @ W
    A = eye - torch.cat([K, torch.zeros_like(K)], 2)
    Cn = A @ C @ A.transpose(1, 2) + K @ V @ K.transpose(1, 2)
    pn = p + (K @ r[:, :, None])[:, :, 0]
    pn = torch.cat([pn[:, :4], torch.remainder(pn[:, 4:5] + math.pi, 2 * math.pi) - math.pi, pn[:, 5:]], 1)
    return torch.where(on[:, None], pn, p), torch.where(on[:, None, None], Cn, C), x2


class _Exact:
    """The geometry and the hits of a batch in FP64."""

    def __init__(self, geom, b):
        d = torch.float64
        self.table = [_dev(geom.kind)] + [_dev(v, d) for v in (geom.pos, geom.lo, geom.hi, geom.x_over_x0)]
        self.kind, self.bz = _dev(geom.kind), float(geom.bz)
        self.xyz, self.cov, self.n_layers = b["xyz"], b["cov"], geom.n_layers
        self.seg_off = _dev(b["seg_off"])

    def layer(self, l):
        return [t[l] for t in self.table]

    def hit(self, h):
        h = h.long().clamp(min=0)
        return self.xyz[h].double(), _tri(self.cov[h].double())

    def fit(self, layers, hits, p0, c0, align=None, xscale=None):
        """Every track through its list; the layers a track fails on end it."""
        p, C = p0.double(), _tri(c0.double())
        sum2 = torch.zeros(len(p), dtype=torch.float64, device=p.device)
        alive = torch.ones(len(p), dtype=torch.bool, device=p.device)
        for j in range(layers.shape[1]):
            on = alive & (layers[:, j] >= 0)
            if not bool(on.any()):
                break
            l = layers[:, j].long().clamp(min=0)
            p, C, ok = _step(p, C, self.layer(l), self.bz, on, xscale=None if xscale is None else xscale[l])
            alive = alive & ~(on & (ok != 1))
            use = on & (ok == 1) & (hits[:, j] >= 0)
            m, V = self.hit(hits[:, j])
            dm = None
            if align is not None:
                c = torch.zeros_like(m)
                c[:, 2] = torch.where(self.kind[l] == 1, self.table[1][l], 0.0)
                dm = align[l, :3] + torch.linalg.cross(align[l, 3:], m - c)
            p, C, x2 = _update(p, C, m, V, use, dm)
            sum2 = sum2 + x2
        return p, C, sum2, alive

    def fit_backward(self, layers, hits, p, C, scale=100.0):
        n = (layers >= 0).sum(1)
        C = C * scale
        sum2 = torch.zeros(len(p), dtype=torch.float64, device=p.device)
        alive = torch.ones(len(p), dtype=torch.bool, device=p.device)
        for j in range(layers.shape[1] - 1, -1, -1):
            l = layers[:, j].long().clamp(min=0)
            first, on = alive & (j == n - 1), alive & (j < n - 1)
            # the start state is taken on its layer: no variance along the surface's normal
            nrm = torch.zeros((len(p), 6), dtype=p.dtype, device=p.device)
            disk, r = self.kind[l] == 1, torch.hypot(p[:, 0], p[:, 1])
            nrm[:, 0], nrm[:, 1] = torch.where(disk, 0.0, p[:, 0] / r), torch.where(disk, 0.0, p[:, 1] / r)
            nrm[:, 2] = torch.where(disk, 1.0, 0.0)
            P = torch.eye(6, dtype=p.dtype, device=p.device) - nrm[:, :, None] * nrm[:, None, :]
            C = torch.where(first[:, None, None], P @ C @ P, C)
            p, C, ok = _step(p, C, self.layer(l), self.bz, on, back=True)
            alive = alive & ~(on & (ok != 1))
            m, V = self.hit(hits[:, j])
            p, C, x2 = _update(p, C, m, V, (first | (on & (ok == 1))) & (hits[:, j] >= 0))
            sum2 = sum2 + x2
        return p, C, sum2

    def seed(self, seeds):
        """Circle through three hits, then a fit through them from a wide prior."""
        hs = [self.hit(seeds[:, j]) for j in range(3)]
        x = [h[0] for h in hs]
        a, b = x[1] - x[0], x[2] - x[0]
        cr = a[:, 0] * b[:, 1] - a[:, 1] * b[:, 0]
        a2, b2 = a[:, 0] ** 2 + a[:, 1] ** 2, b[:, 0] ** 2 + b[:, 1] ** 2
        line = cr.abs() < 1e-12 * b2
        crs = torch.where(line, 1.0, cr)
        ux, uy = (b[:, 1] * a2 - a[:, 1] * b2) / (2 * crs), (a[:, 0] * b2 - b[:, 0] * a2) / (2 * crs)
        rho, sg = torch.hypot(ux, uy), torch.sign(crs)
        vx, vy = b[:, 0] - ux, b[:, 1] - uy
        turn = torch.atan2(-ux * vy + uy * vx, -ux * vx - uy * vy).abs()
        arc = torch.where(line, torch.sqrt(b2), turn * rho)
        k = torch.where(line, 1e-12, -sg / (rho * C_LIGHT * self.bz))
        phi = torch.where(line, torch.atan2(b[:, 1], b[:, 0]), torch.atan2(-sg * ux, sg * uy))
        th = torch.atan2(torch.ones_like(arc), b[:, 2] / arc)
        p = torch.cat([x[0], torch.stack([k, phi, th], 1)], 1)
        sk = 0.5 * k.abs() + 0.05
        w = torch.full((len(p), 6), 0.01, dtype=p.dtype, device=p.device)
        w[:, 3], w[:, 4], w[:, 5] = sk * sk, 0.0025, 0.0025
        C = torch.diag_embed(w)
        on = torch.ones(len(p), dtype=torch.bool, device=p.device)
        p, C, _ = _update(p, C, *hs[0], on)
        for j in (1, 2):
            seg = torch.bucketize(seeds[:, j].long(), self.seg_off[1:], right=True)
            p, C, ok = _step(p, C, self.layer(seg % self.n_layers), self.bz, on)
            on = on & (ok == 1)
            p, C, _ = _update(p, C, *hs[j], on)
        return p, C


def _chunks(n, size):
    return [slice(i, min(n, i + size)) for i in range(0, n, size)]


def exact(case, seed):
    call = case["call"]
    if call in ("modular", "clean"):   # planes: no plain reference here; whole numbers
        return None
    geom, b = _make(case, seed)
    ex = _Exact(geom, b)
    none_tracks = dict.fromkeys(("params", "cov", "chi2", "score", "nfound", "nholes", "hits"))
    if call == "seed":
        parts = [ex.seed(b["seeds"][q]) for q in _chunks(len(b["seeds"]), 200_000)]
        return {"state": torch.cat([p for p, _ in parts]), "cov": torch.cat([_pack(C) for _, C in parts]), "info": None}
    layers, hits, p0, c0 = (b[k] for k in ("layers", "hits", "p0", "c0"))
    if call == "grad":
        al, xs = b["align"].double().requires_grad_(), b["xscale"].double().requires_grad_()
        total, gp = 0.0, []
        for q in _chunks(len(p0), 8_000):
            pq = p0[q].double().requires_grad_()
            _, _, x2, alive = ex.fit(layers[q], hits[q], pq, c0[q], al, xs)
            t = torch.where(alive, x2, 0.0).sum()
            t.backward()
            total += float(t)
            gp.append(pq.grad)
        return {"chi2": total, "align": al.grad, "xscale": xs.grad, "p0": torch.cat(gp), "status": None}
    if call == "backward":
        layers, hits = _outer(layers), _outer(hits)
    fits, backs = [], []
    for q in _chunks(len(p0), 200_000):
        p, C, x2, _ = ex.fit(layers[q], hits[q], p0[q], c0[q])
        fits.append((p, _pack(C), x2))
        if call == "backward":
            p, C, x2 = ex.fit_backward(layers[q], hits[q], p, C)
            backs.append((p, _pack(C), x2))
    whole = lambda parts: dict(zip(("p", "c", "chi2"), (torch.cat(v) for v in zip(*parts))), status=None)
    if call == "fit":
        return {"fit": whole(fits)}
    if call == "backward":
        return {"fit": whole(fits), "back": whole(backs), "tracks": none_tracks}
    return {"tracks": none_tracks, "fit": whole(fits)}
