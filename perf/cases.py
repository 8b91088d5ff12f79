"""What a user of this library has it do, as cases that can be timed and compared.

Each case is a dict of plain values.  ``prepare`` makes what a user's program
holds before the call (data, plan, template bank), ``run`` is one pass through
the public entry points, ``work`` says what that pass cannot do without and
``exact`` gives the same result from plain torch in 64 bits.

Kinds:
  dense   2F of every bin for a bank of templates (fstat_compute); every pass
          redoes the per-sky work, as a search over sky positions does
  peaks   the same bank reduced on the device to band maxima and the list of
          2F > 70 (fstat_compute_peaks), read back by the host
  batch   uneven targets replayed as one CUDA graph (fstat_batch_*)
  semi    semi-coherent sum over data segments, then its peaks reduction
  grad    2F and its gradient at refinement candidates (fstat_grad)
  sft     short Fourier transforms in host memory -> series -> 2F
  noalloc one template from a caller's resampled series (fstat_twoF_noalloc)
"""

import ctypes
import math
from types import SimpleNamespace

import numpy as np
import torch

import paper_2201_00451_gb300 as fs

DAY = 86400.0
TWO_PI = 2.0 * math.pi
THRESHOLD = 70.0
CAPACITY = 4096  # of the crossing list
EPHEMERIS = {
    "c": 299792458.0, "au": 1.495978707e11, "r_earth": 6.371e6,
    "omega_rot": TWO_PI / 86164.0905, "omega_orb": TWO_PI / (365.25636 * DAY),
    "obliquity": math.radians(23.4393), "orb_phase0": 0.0, "sidereal_phase0": 0.0,
}
SITES = tuple(SimpleNamespace(lat=math.radians(a), lon=math.radians(b), gamma=math.radians(c))
              for a, b, c in ((46.455, -119.408, 171.8), (30.563, -90.774, 243.0)))


# ------------------------------------------------------------------- the cases
def listed():
    return [
        # a first look at a short stretch of data: a ragged series and a handful
        # of spindowns, where launches and latency count
        {"name": "short_look_2e13", "kind": "dense", "n": 3001, "dt": 2.0, "n_fft": 1 << 13, "det": 2, "sky": 1,
         "f1": 4, "f2": 1, "dterms": 8, "interp": 0, "fp64": False, "c128": False, "tune": False, "f_het": 100.0},
        # one template inside a host application that owns the memory pool
        {"name": "plug_in_2e18", "kind": "noalloc", "n": 86400, "dt": 2.0, "n_fft": 1 << 18},
        # the plain method: FP64 throughout, 2 days, 64 spindowns
        {"name": "plain_fp64_2e18", "kind": "dense", "n": 86400, "dt": 2.0, "n_fft": 1 << 18, "det": 1, "sky": 1,
         "f1": 64, "f2": 1, "dterms": 8, "interp": 0, "fp64": True, "c128": True, "tune": False, "f_het": 100.0},
        # a few sky positions of a medium data set with a wider, untapered
        # interpolator, without tuning: an odd length, a third of a week
        {"name": "medium_2e19", "kind": "dense", "n": 400001, "dt": 1.0, "n_fft": 1 << 19, "det": 2, "sky": 3,
         "f1": 8, "f2": 1, "dterms": 16, "interp": 1, "fp64": False, "c128": False, "tune": False, "f_het": 212.5},
        # follow-up of uneven targets (1 to 30 days, 0.5 to 4 Hz) in one graph
        {"name": "uneven_targets", "kind": "batch",
         "targets": "1036800 0.25 2097152 32 241.3;86400 1.0 262144 128 294.7;1296000 2.0 4194304 32 318.4"},
        # the 10-day narrowband search of one target, a slice of its bank
        {"name": "narrow_2e22", "kind": "dense", "n": 1728000, "dt": 0.5, "n_fft": 1 << 22, "det": 2, "sky": 1,
         "f1": 32, "f2": 2, "dterms": 8, "interp": 0, "fp64": False, "c128": False, "tune": True, "f_het": 100.0},
        # many sky positions with few spindowns each (the pilot search's shape)
        {"name": "many_skies_2e22", "kind": "dense", "n": 1728000, "dt": 0.5, "n_fft": 1 << 22, "det": 2, "sky": 6,
         "f1": 11, "f2": 1, "dterms": 8, "interp": 0, "fp64": False, "c128": False, "tune": True, "f_het": 100.0},
        # the 120-day search with every bin kept
        {"name": "large_2e24", "kind": "dense", "n": 10368000, "dt": 1.0, "n_fft": 1 << 24, "det": 2, "sky": 1,
         "f1": 12, "f2": 2, "dterms": 8, "interp": 0, "fp64": False, "c128": False, "tune": True, "f_het": 217.25},
        # the 120-day search reduced on the device, as the search proper runs it
        {"name": "large_peaks_2e24", "kind": "peaks", "n": 10368000, "dt": 1.0, "n_fft": 1 << 24, "det": 2, "sky": 1,
         "f1": 8, "f2": 2, "dterms": 8, "interp": 0, "fp64": False, "c128": False, "tune": True, "f_het": 217.25,
         "bands": 32},
        # ten-day segments summed semi-coherently, then reduced
        {"name": "segments_2e22", "kind": "semi", "n": 1728000, "dt": 0.5, "n_fft": 1 << 22, "det": 2, "segs": 4,
         "f1": 6, "f2": 1, "f_het": 100.0, "tune": True, "bands": 16},
        # off-grid follow-up of candidates of the 10-day search
        {"name": "candidates_10d", "kind": "grad", "n": 1728000, "dt": 0.5, "det": 2, "cand": 256, "f_het": 100.0,
         "fp64": False, "c128": False},
        # from SFT bins on the host (480 half-hour SFTs, 2 Hz) to 2F
        {"name": "sfts_10d", "kind": "sft", "n_sft": 480, "n_bins": 3600, "t_sft": 1800.0, "n_fft": 1 << 22, "det": 2,
         "f1": 2, "f2": 1, "fp64": False, "c128": False},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _samples(rng, n_fft):
    """An odd or ragged series length that is padded to n_fft."""
    return max(1000, int(n_fft * rng.uniform(0.26, 0.98))) | rng.randrange(2)


def _detectors(rng, span):
    """One detector alone needs half a day to tell the two polarisations apart."""
    return rng.choice((1, 2, 2)) if span >= 0.5 * DAY else 2


def draw(rng):
    kind = rng.choice(("dense", "dense", "dense", "peaks", "batch", "semi", "grad", "sft", "noalloc"))
    if kind == "dense":
        fp64 = rng.random() < 0.2
        n_fft = 1 << rng.randint(13, 20 if fp64 else 24)
        sky = rng.choice((1, 1, 2, 3, 5))
        most = (1 << 24 if fp64 else 24 << 24) // (n_fft * sky)
        f1 = max(1, min(_log_int(rng, 2, 96), most))
        n, dt = _samples(rng, n_fft), rng.choice((0.25, 0.5, 1.0, 2.0))
        return {"kind": kind, "n": n, "dt": dt, "n_fft": n_fft, "det": _detectors(rng, n * dt),
                "sky": sky, "f1": f1, "f2": 2 if 2 * f1 <= min(most, 64) else 1,
                "dterms": rng.choice((4, 8, 8, 8, 16, 32)), "interp": rng.choice((0, 0, 1, 2)), "fp64": fp64,
                "c128": fp64 or rng.random() < 0.2, "tune": rng.random() < 0.5, "f_het": rng.uniform(100.0, 490.0)}
    if kind == "peaks":
        n_fft = 1 << rng.randint(18, 24)
        f1 = max(1, min(_log_int(rng, 4, 48), (16 << 24) // n_fft))
        n, dt = _samples(rng, n_fft), rng.choice((0.5, 1.0, 2.0))
        return {"kind": kind, "n": n, "dt": dt, "n_fft": n_fft, "det": _detectors(rng, n * dt),
                "sky": 1, "f1": f1, "f2": 1, "dterms": 8, "interp": 0, "fp64": False, "c128": False,
                "tune": rng.random() < 0.5, "f_het": rng.uniform(100.0, 490.0),
                "bands": rng.choice((1, 4, 16))}
    if kind == "batch":
        parts = []
        for _ in range(rng.randint(2, 4)):
            n_fft = 1 << rng.randint(18, 22)
            t = max(4, min(_log_int(rng, 8, 128), (64 << 22) // n_fft))
            parts.append("%d %g %d %d %.3f" % (_samples(rng, n_fft), rng.choice((0.25, 0.5, 1.0, 2.0)), n_fft, t,
                                               rng.uniform(145.0, 490.0)))
        return {"kind": kind, "targets": ";".join(parts)}
    if kind == "semi":
        n_fft = 1 << rng.randint(16, 22)
        n, dt = _samples(rng, n_fft), rng.choice((0.5, 1.0, 2.0))
        return {"kind": kind, "n": n, "dt": dt, "n_fft": n_fft, "det": _detectors(rng, n * dt),
                "segs": rng.randint(2, 6), "f1": rng.randint(2, 8), "f2": 1,
                "f_het": rng.uniform(100.0, 490.0), "tune": rng.random() < 0.5, "bands": rng.choice((1, 4, 16))}
    if kind == "grad":
        n, dt = _log_int(rng, 20000, 1728000) | 1, rng.choice((0.25, 0.5, 1.0, 2.0))
        return {"kind": kind, "n": n, "dt": dt, "det": _detectors(rng, n * dt),
                "cand": _log_int(rng, 1, 300), "f_het": rng.uniform(100.0, 490.0), "fp64": False,
                "c128": rng.random() < 0.2}
    if kind == "sft":
        bins = rng.choice((900, 1800, 3600, 90 * rng.randint(4, 60), rng.randint(300, 4200)))
        n_sft = _log_int(rng, 8, 480)
        n_fft = 1 << max(13, (n_sft * bins - 1).bit_length())
        t_sft = rng.choice((900.0, 1800.0))
        return {"kind": kind, "n_sft": n_sft, "n_bins": bins, "t_sft": t_sft, "n_fft": n_fft,
                "det": _detectors(rng, n_sft * t_sft), "f1": rng.randint(1, 4), "f2": 1, "fp64": False,
                "c128": rng.random() < 0.2}
    n_fft = 1 << rng.randint(10, 18)
    return {"kind": kind, "n": max(500, int(n_fft * rng.uniform(0.3, 0.98))) | rng.randrange(2),
            "dt": rng.choice((0.5, 1.0, 2.0)), "n_fft": n_fft}


# ------------------------------------------------------- timing model in 64 bits
def _sky_vector(alpha, delta):
    return (math.cos(delta) * math.cos(alpha), math.cos(delta) * math.sin(alpha), math.sin(delta))


def _position(t, site):
    """Detector position over c (seconds) at times t: three tensors."""
    e = EPHEMERIS
    th = e["orb_phase0"] + e["omega_orb"] * t
    ph = site.lon + e["sidereal_phase0"] + e["omega_rot"] * t
    rc, rs = e["r_earth"] * math.cos(site.lat), e["r_earth"] * math.sin(site.lat)
    so = torch.sin(th)
    return ((e["au"] * torch.cos(th) + rc * torch.cos(ph)) / e["c"],
            (e["au"] * math.cos(e["obliquity"]) * so + rc * torch.sin(ph)) / e["c"],
            (e["au"] * math.sin(e["obliquity"]) * so + rs) / e["c"])


def _delay(t, site, alpha, delta):
    n, r = _sky_vector(alpha, delta), _position(t, site)
    return r[0] * n[0] + r[1] * n[1] + r[2] * n[2]


def _tensor(t, site):
    """Detector tensor (xx, yy, zz, xy, xz, yz) at times t."""
    ph = site.lon + EPHEMERIS["sidereal_phase0"] + EPHEMERIS["omega_rot"] * t
    c, s = torch.cos(ph), torch.sin(ph)
    sl, cl = math.sin(site.lat), math.cos(site.lat)
    east = (-s, c, torch.zeros_like(s))
    north = (-sl * c, -sl * s, cl * torch.ones_like(s))
    g = (site.gamma - math.pi / 4, site.gamma + math.pi / 4)
    u, v = ([math.cos(a) * east[i] + math.sin(a) * north[i] for i in range(3)] for a in g)
    return [0.5 * (u[p] * u[q] - v[p] * v[q]) for p, q in ((0, 0), (1, 1), (2, 2), (0, 1), (0, 2), (1, 2))]


def _polarisation(alpha, delta):
    """e+ and ex on (xx, yy, zz, xy, xz, yz), off-diagonals doubled, and their sky derivatives."""
    sa, ca, sd, cd = math.sin(alpha), math.cos(alpha), math.sin(delta), math.cos(delta)
    x, y = (sa, -ca, 0.0), (-sd * ca, -sd * sa, cd)
    xa, ya = (ca, sa, 0.0), (sd * sa, -sd * ca, 0.0)
    xd, yd = (0.0, 0.0, 0.0), (-cd * ca, -cd * sa, -sd)
    pq = ((0, 0, 1.0), (1, 1, 1.0), (2, 2, 1.0), (0, 1, 2.0), (0, 2, 2.0), (1, 2, 2.0))

    def plus(u, v, uu, vv):
        return [w * (u[p] * uu[q] + uu[p] * u[q] - v[p] * vv[q] - vv[p] * v[q]) for p, q, w in pq]

    def cross(u, v, uu, vv):
        return [w * (uu[p] * v[q] + v[p] * uu[q] + u[p] * vv[q] + vv[p] * u[q]) for p, q, w in pq]

    half = [[0.5 * k for k in e] for e in (plus(x, y, x, y), cross(x, y, x, y))]
    return half, (plus(x, y, xa, ya), cross(x, y, xa, ya)), (plus(x, y, xd, yd), cross(x, y, xd, yd))


def _contract(d, e):
    return sum(d[k] * e[k] for k in range(6))


def _antenna(t, site, alpha, delta):
    d = _tensor(t, site)
    (ep, ex), _, _ = _polarisation(alpha, delta)
    return _contract(d, ep), _contract(d, ex)


def _turns(phase):
    """exp(2 pi i phase) for a phase in cycles."""
    return torch.polar(torch.ones_like(phase), TWO_PI * (phase - torch.floor(phase)))


def _times(c, t0=0.0):
    return t0 + torch.arange(c["n"], dtype=torch.float64, device="cuda") * c["dt"]


# ------------------------------------------------------------------- the inputs
def _rng(seed, sub=0):
    return np.random.Generator(np.random.PCG64(np.random.SeedSequence([int(seed), sub])))


def _spans(n, dt):
    t = n * dt
    return 1.0 / (4.0 * t * t), 1.0 / (8.0 * t ** 3)


def _bank(rng, c):
    """Template bank: a patch of sky positions x a spindown grid."""
    a0, d0 = rng.uniform(0.0, TWO_PI), math.asin(rng.uniform(-0.95, 0.95))
    s1, s2 = _spans(c["n"], c["dt"])
    arcmin = math.radians(1.0 / 60.0)
    sky = [(a0 + k * arcmin / 8.0 / math.cos(d0), d0 + (k % 3) * arcmin / 8.0) for k in range(c.get("sky", 1))]
    rows = [(a, d, -s1 * (c["f1"] - 1 - i), s2 * (j - 0.5 * (c["f2"] - 1)))
            for a, d in sky for j in range(c["f2"]) for i in range(c["f1"])]
    return fs.as_templates(np.array(rows))


def _signals(c, seed, bank, n_fft, sub=0):
    """Two signals on templates of the bank, at bins of the inner band."""
    rng = _rng(seed, 1000 + sub)
    out = []
    for _ in range(2):
        cosi, psi = rng.uniform(-1, 1), rng.uniform(-0.78, 0.78)
        ap = 0.5 * (1 + cosi * cosi)
        out.append(SimpleNamespace(
            tm=bank[int(rng.integers(len(bank)))], rho2=rng.uniform(100, 300), phi0=rng.uniform(0, 1),
            off=int(rng.integers(-int(0.4 * n_fft), int(0.4 * n_fft))) / (n_fft * c["dt"]),
            ka=complex(ap * math.cos(2 * psi), cosi * math.sin(2 * psi)) / 2,
            kb=complex(ap * math.sin(2 * psi), -cosi * math.cos(2 * psi)) / 2))
    return out


def _fft_length(c):
    return c.get("n_fft", 1 << max(10, (c["n"] - 1).bit_length()))


def _series(c, seed, bank, t0=0.0, sub=0):
    """Per detector: seeded noise with two signals of the bank, and the noise levels."""
    sigmas = [float(s) for s in _rng(seed, 1 + sub).uniform(0.8, 1.2, c["det"])]
    g = torch.Generator(device="cuda").manual_seed(1000003 * (int(seed) % (1 << 40)) + sub)
    xs = []
    for s in sigmas:
        v = torch.randn((c["n"], 2), generator=g, device="cuda", dtype=torch.float64 if c.get("c128") else torch.float32)
        xs.append(torch.view_as_complex(v * s))
    t, t_ref = _times(c, t0), t0 + (c["n"] // 2) * c["dt"]
    for q in _signals(c, seed, bank, _fft_length(c), sub):
        sky, parts, power = (float(q.tm["alpha"]), float(q.tm["delta"])), [], 0.0
        for X in range(c["det"]):
            tm = _delay(t, SITES[X], *sky)
            a, b = _antenna(t, SITES[X], *sky)
            tau = t + tm - t_ref
            ph = (q.off * tau + torch.frac(c["f_het"] * tm) + float(q.tm["f1dot"]) * tau * tau / 2
                  + float(q.tm["f2dot"]) * tau ** 3 / 6)
            parts.append((q.ka * a + q.kb * b) * _turns(ph + q.phi0))
            power = power + (parts[-1].abs() ** 2).sum() / sigmas[X] ** 2
        for X, p in enumerate(parts):
            xs[X] += (torch.sqrt(q.rho2 / power) * p).to(xs[X].dtype)
    return xs, sigmas


def _plan(c, xs, sigmas, t0=0.0):
    plan = fs.FstatPlan(fs.make_desc(
        detectors=SITES[:c["det"]], t0=t0, dt=c["dt"], n_samples=c["n"], f_het=c["f_het"], n_fft=_fft_length(c),
        dterms=c.get("dterms", 8), precision=fs.FP64 if c.get("fp64") else fs.MIXED, ephemeris=EPHEMERIS,
        interp=c.get("interp", 0)))
    for X, x in enumerate(xs):
        plan.set_data(X, x, sigmas[X])
    if c.get("tune"):
        plan.autotune()
    return plan


def _targets(c):
    """The targets of a batch case as dense cases of their own."""
    out = []
    for part in c["targets"].split(";"):
        n, dt, n_fft, f1, f_het = part.split()
        out.append({"n": int(n), "dt": float(dt), "n_fft": int(n_fft), "f1": int(f1), "f2": 1, "det": 2,
                    "f_het": float(f_het), "tune": True})
    return out


def _segments(c, seed):
    bank = _bank(_rng(seed), dict(c, n=c["n"] * c["segs"]))
    parts = []
    for s in range(c["segs"]):
        t0 = s * c["n"] * c["dt"]
        parts.append((t0,) + _series(c, seed, bank, t0, 10 * s))
    return bank, 0.5 * c["segs"] * c["n"] * c["dt"], parts


def _candidates(c, seed):
    """Candidates within half a grid step of the signals, as a search hands them on."""
    rng = _rng(seed, 2)
    bank = _bank(_rng(seed), dict(c, f1=64, f2=1))
    found = _signals(c, seed, bank, _fft_length(c))
    s1, s2 = _spans(c["n"], c["dt"])
    out = np.zeros(c["cand"], dtype=fs.CANDIDATE_DTYPE)
    for i in range(c["cand"]):
        q = found[i % 2]
        out[i] = (c["f_het"] + q.off + rng.uniform(-0.5, 0.5) / (c["n"] * c["dt"]), q.tm["f1dot"] + s1 * rng.uniform(-0.5, 0.5),
                  q.tm["alpha"] + rng.uniform(-1e-5, 1e-5), q.tm["delta"] + rng.uniform(-1e-5, 1e-5), s2 * rng.uniform(-2, 2))
    return bank, out


def _sfts(c, seed):
    """SFT bins per detector in host memory (pinned, as a reader's buffers are), of unit noise."""
    full = dict(c, n=c["n_sft"] * c["n_bins"], dt=c["t_sft"] / c["n_bins"], f_het=100.0)
    bank = _bank(_rng(seed), full)
    g = torch.Generator(device="cuda").manual_seed(7 + 1000003 * (int(seed) % (1 << 40)))
    m_raw = 2 * c["n_bins"]
    bins = []
    for _ in range(c["det"]):
        v = torch.randn((c["n_sft"], c["n_bins"], 2), generator=g, device="cuda",
                        dtype=torch.float64 if c["c128"] else torch.float32)
        bins.append(torch.view_as_complex(v * (m_raw / math.sqrt(c["n_bins"]))))
    return full, bank, bins, m_raw


def _resampled(c, seed):
    """A caller's own resampled series: unit noise under two slow patterns, and their A, B, C."""
    rng = _rng(seed)
    g = torch.Generator(device="cuda").manual_seed(13 + 1000003 * (int(seed) % (1 << 40)))
    t = _times(c)
    p = rng.uniform(0.1, 0.5, 4)
    w = TWO_PI * rng.uniform(0.8, 3.0) / (c["n"] * c["dt"])
    a = p[0] + p[1] * torch.cos(2 * w * t + rng.uniform(0, 6))
    b = p[2] * torch.sin(w * t + rng.uniform(0, 6)) + p[3]
    v = torch.randn((c["n"], 2), generator=g, device="cuda", dtype=torch.float64)
    pairs = torch.cat((0.5 * a[:, None] * v, 0.5 * b[:, None] * v), 1).float().contiguous()
    abc = [float(0.5 * (x * y).sum()) for x, y in ((a, a), (b, b), (a, b))]
    s1, s2 = _spans(c["n"], c["dt"])
    return pairs, abc, -(c["n"] // 2) * c["dt"], -s1 * rng.uniform(0, 50), s2 * rng.uniform(-2, 2)


def prepare(case, seed):
    c, s = case, SimpleNamespace(case=case)
    if c["kind"] in ("dense", "peaks"):
        s.bank = _bank(_rng(seed), c)
        s.plan = _plan(c, *_series(c, seed, s.bank))
        if c["kind"] == "dense":
            s.out = torch.empty((len(s.bank), c["n_fft"]), dtype=torch.float32, device="cuda")
    elif c["kind"] == "batch":
        s.plans, s.outs, s.batch = [], [], fs.FstatBatch()
        for k, t in enumerate(_targets(c)):
            bank = _bank(_rng(seed, 100 + k), t)
            s.plans.append(_plan(t, *_series(t, seed, bank, sub=k)))
            s.outs.append(torch.empty((len(bank), t["n_fft"]), dtype=torch.float32, device="cuda"))
            s.batch.add(s.plans[-1], bank, s.outs[-1])
        s.batch.instantiate()
    elif c["kind"] == "semi":
        s.bank, s.t_ref, parts = _segments(c, seed)
        s.plans = [_plan(c, xs, sigmas, t0) for t0, xs, sigmas in parts]
        s.out = torch.empty((len(s.bank), c["n_fft"]), dtype=torch.float32, device="cuda")
    elif c["kind"] == "grad":
        bank, s.cand = _candidates(c, seed)
        s.plan = _plan(c, *_series(c, seed, bank))
    elif c["kind"] == "sft":
        s.full, s.bank, bins, s.m_raw = _sfts(c, seed)
        s.host = [torch.empty(b.shape, dtype=b.dtype, pin_memory=True).copy_(b) for b in bins]
        s.bins = [h.numpy() for h in s.host]
        s.plan = _plan(s.full, [], [])
        s.out = torch.empty((len(s.bank), c["n_fft"]), dtype=torch.float32, device="cuda")
    else:
        s.pairs, s.abc, s.tau0, s.f1dot, s.f2dot = _resampled(c, seed)
        s.out = torch.empty(c["n_fft"], dtype=torch.float32, device="cuda")
    return s


# -------------------------------------------------------------------- one pass
def run(s):
    c = s.case
    if c["kind"] == "dense":
        s.plan.invalidate_sky()
        return s.plan.compute(s.bank, out=s.out)
    if c["kind"] == "peaks":
        s.plan.invalidate_sky()
        r = s.plan.compute_peaks(s.bank, threshold=THRESHOLD, n_bands=c["bands"], capacity=CAPACITY)
        found = fs.peaks_to_numpy(r)  # the list comes in no order
        table = np.zeros(CAPACITY, dtype=found.dtype)
        table[:len(found)] = found[np.lexsort((found["bin"], found["tmpl"]))]
        return {"count": r["count"], "band_max": r["band_max"], "band_bin": r["band_bin"],
                "tmpl": table["tmpl"], "bin": table["bin"], "twoF": table["twoF"]}
    if c["kind"] == "batch":
        s.batch.launch()
        return s.outs
    if c["kind"] == "semi":
        for p in s.plans:
            p.invalidate_sky()
        fs.semicoherent(s.plans, s.bank, s.t_ref, out=s.out)
        r = s.plans[0].reduce_peaks(s.out, threshold=1e30, n_bands=c["bands"])
        return {"sum": s.out, "band_max": r["band_max"], "band_bin": r["band_bin"]}
    if c["kind"] == "grad":
        two_f, g = s.plan.grad(s.cand)
        return {"twoF": two_f, "grad": g}
    if c["kind"] == "sft":
        for X, b in enumerate(s.bins):
            s.plan.set_sfts(X, b, int(round(100.0 * c["t_sft"])) - c["n_bins"] // 2, c["t_sft"], s.m_raw, 1.0)
        return s.plan.compute(s.bank, out=s.out)
    rc = fs.load().fstat_twoF_noalloc(
        ctypes.c_void_p(s.pairs.data_ptr()), c["n"], c["n_fft"], c["dt"], s.tau0, s.abc[0], s.abc[1], s.abc[2],
        s.f1dot, s.f2dot, ctypes.c_void_p(s.out.data_ptr()),
        ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    if rc != fs.OK:
        raise fs.FstatError(rc, "fstat_twoF_noalloc")
    return s.out


# ------------------------------------------------------------------------ work
def _dense_work(c, skies, n_tmpl, elem, written):
    fft = 10.0 * c["n_fft"] * math.log2(c["n_fft"])  # two complex transforms
    per_sky = c["det"] * c["n"] * (4.0 * (2 * c.get("dterms", 8) + 1) + 20.0)
    return {"bytes": float(skies * c["det"] * c["n"] * elem + n_tmpl * written),
            "flops": skies * per_sky + n_tmpl * (fft + 12.0 * c["n"] + 12.0 * c["n_fft"])}


def work(case):
    c = case
    elem = 16 if c.get("c128") else 8
    if c["kind"] == "dense":
        return _dense_work(c, 1, c["sky"] * c["f1"] * c["f2"], elem, 4 * c["n_fft"])
    if c["kind"] == "peaks":
        return _dense_work(c, 1, c["f1"] * c["f2"], elem, 8 * c["bands"])
    if c["kind"] == "batch":
        parts = [_dense_work(t, 1, t["f1"], 8, 4 * t["n_fft"]) for t in _targets(c)]
        return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}
    if c["kind"] == "semi":
        one = _dense_work(c, 1, c["f1"] * c["f2"], 8, 0)
        return {"bytes": c["segs"] * one["bytes"] + 4.0 * c["f1"] * c["f2"] * c["n_fft"], "flops": c["segs"] * one["flops"]}
    if c["kind"] == "grad":
        # per candidate and sample: a phase, its rotation, and the products
        # that enter Fa, Fb and their four derivatives
        return {"bytes": float(c["det"] * c["n"] * elem + 60 * c["cand"]), "flops": 60.0 * c["cand"] * c["det"] * c["n"]}
    if c["kind"] == "sft":
        n = c["n_sft"] * c["n_bins"]
        full = _dense_work(dict(c, n=n), 1, c["f1"] * c["f2"], elem, 4 * c["n_fft"])
        return {"bytes": full["bytes"], "flops": full["flops"] + c["det"] * 5.0 * n * math.log2(c["n_bins"])}
    return {"bytes": 16.0 * c["n"] + 4.0 * c["n_fft"], "flops": 10.0 * c["n_fft"] * math.log2(c["n_fft"])}


# --------------------------------------------------------- the result in 64 bits
def _weight(x, n, d, kind):
    one = x == 0
    x = torch.where(one, torch.full_like(x, 0.5), x)
    m = 2 * d + 1 if kind == 2 else n
    w = torch.sin(math.pi * x) / (m * torch.sin(math.pi * x / m))
    if kind == 0:
        w = w * (0.54 + 0.46 * torch.cos(math.pi * x / (d + 1)))
    return torch.where(one, torch.ones_like(w), w)


def _exact_sky(c, xs, sigmas, alpha, delta, t0):
    """Ga, Gb, A, B, C and the first SSB epoch of one sky position."""
    n, d, kind = c["n"], c.get("dterms", 8), c.get("interp", 0)
    t = _times(c, t0)
    e, nv = EPHEMERIS, _sky_vector(alpha, delta)
    th = e["orb_phase0"] + e["omega_orb"] * (t0 + 0.5 * n * c["dt"])
    orb = e["au"] * (math.cos(th) * nv[0] + math.sin(th) * (math.cos(e["obliquity"]) * nv[1] + math.sin(e["obliquity"]) * nv[2]))
    tb = (t0 + orb / e["c"]) + torch.arange(n, dtype=torch.float64, device="cuda") * c["dt"]
    ga = torch.zeros(n, dtype=torch.complex128, device="cuda")
    gb, abc = torch.zeros_like(ga), [0.0, 0.0, 0.0]
    for X, x in enumerate(xs):
        w = 0.5 / sigmas[X] ** 2
        z = x.to(torch.complex128) * _turns(-c["f_het"] * _delay(t, SITES[X], alpha, delta))
        T = tb - _delay(tb, SITES[X], alpha, delta)
        for _ in range(3):
            T = tb - _delay(T, SITES[X], alpha, delta)
        u = (T - t0) / c["dt"]
        k0 = torch.round(u)
        frac = u - k0
        k0 = k0.long()
        valid = (k0 >= 0) & (k0 <= n - 1)
        zi = torch.zeros_like(ga)
        for m in range(-d, d + 1):
            k = k0 + m
            ok = valid & (k >= 0) & (k < n)
            zi += torch.where(ok, z[k.clamp(0, n - 1)] * _weight(frac - m, n, d, kind), 0.0)
        a, b = _antenna(T, SITES[X], alpha, delta)
        a, b = torch.where(valid, a, 0.0), torch.where(valid, b, 0.0)
        ga += w * a * zi
        gb += w * b * zi
        abc = [v + w * float((p * q).sum()) for v, (p, q) in zip(abc, ((a, a), (b, b), (a, b)))]
    return ga, gb, abc, float(tb[0])


def _exact_row(ga, gb, abc, tau, f1dot, f2dot, n_fft):
    rot = _turns(-(f1dot * tau * tau / 2 + f2dot * tau * tau * tau / 6))
    fa, fb = (torch.fft.fftshift(torch.fft.fft(g * rot, n=n_fft)) for g in (ga, gb))
    A, B, C = abc
    return 2.0 * (B * fa.abs() ** 2 + A * fb.abs() ** 2 - 2.0 * C * (fa * fb.conj()).real) / (A * B - C * C)


def _exact_rows(c, xs, sigmas, bank, t0=0.0):
    key, prep = None, None
    for tm in bank:
        if (float(tm["alpha"]), float(tm["delta"])) != key:
            key = (float(tm["alpha"]), float(tm["delta"]))
            prep = _exact_sky(c, xs, sigmas, key[0], key[1], t0)
        ga, gb, abc, tb0 = prep
        tau = tb0 + torch.arange(c["n"], dtype=torch.float64, device="cuda") * c["dt"] - (t0 + (c["n"] // 2) * c["dt"])
        yield _exact_row(ga, gb, abc, tau, float(tm["f1dot"]), float(tm["f2dot"]), c["n_fft"])


def _exact_grad(c, xs, sigmas, cand):
    t_ref = (c["n"] // 2) * c["dt"]
    t = _times(c)
    two_f, grad = np.empty(len(cand)), np.empty((len(cand), 4))
    sites = [(0.5 / sigmas[X] ** 2, x.to(torch.complex128), _position(t, SITES[X]), _tensor(t, SITES[X]))
             for X, x in enumerate(xs)]
    for i, q in enumerate(cand):
        f, f1, al, de, f2 = (float(q[k]) for k in ("f", "f1dot", "alpha", "delta", "f2dot"))
        n, na, nd = _sky_vector(al, de), (-math.cos(de) * math.sin(al), math.cos(de) * math.cos(al), 0.0), \
            (-math.sin(de) * math.cos(al), -math.sin(de) * math.sin(al), math.cos(de))
        e0, ea, ed = _polarisation(al, de)
        F = np.zeros((5, 2), dtype=complex)  # value, d/df, d/df1dot, d/dalpha, d/ddelta
        S = np.zeros((3, 3))                 # A, B, C: value, d/dalpha, d/ddelta
        for w, x, r, d in sites:
            tm = r[0] * n[0] + r[1] * n[1] + r[2] * n[2]
            tau = t + tm - t_ref
            ph = (f - c["f_het"]) * tau + torch.frac(c["f_het"] * tm) + f1 * tau * tau / 2 + f2 * tau ** 3 / 6
            e = w * x * _turns(-ph)
            pat = [[_contract(d, p[k]) for k in (0, 1)] for p in (e0, ea, ed)]
            rate = f + f1 * tau + 0.5 * f2 * tau * tau
            dphi = [tau, 0.5 * tau * tau] + [rate * (r[0] * v[0] + r[1] * v[1] + r[2] * v[2]) for v in (na, nd)]
            for k in (0, 1):
                ek = e * pat[0][k]
                F[0, k] += complex(ek.sum())
                for j in range(4):
                    F[1 + j, k] += -1j * TWO_PI * complex((ek * dphi[j]).sum())
                F[3, k] += complex((e * pat[1][k]).sum())
                F[4, k] += complex((e * pat[2][k]).sum())
            for row, (u, v) in enumerate(((0, 0), (1, 1), (0, 1))):
                S[row, 0] += w * float((pat[0][u] * pat[0][v]).sum())
                for j in (1, 2):
                    S[row, j] += w * float((pat[j][u] * pat[0][v] + pat[0][u] * pat[j][v]).sum())
        A, B, C = S[:, 0]
        D = A * B - C * C
        N = B * abs(F[0, 0]) ** 2 + A * abs(F[0, 1]) ** 2 - 2 * C * (F[0, 0] * F[0, 1].conjugate()).real
        two_f[i] = 2 * N / D
        for j in range(4):
            fa, fb = F[1 + j]
            dA, dB, dC = S[:, j - 1] if j >= 2 else (0.0, 0.0, 0.0)
            dN = (dB * abs(F[0, 0]) ** 2 + dA * abs(F[0, 1]) ** 2
                  + 2 * B * (F[0, 0].conjugate() * fa).real + 2 * A * (F[0, 1].conjugate() * fb).real
                  - 2 * dC * (F[0, 0] * F[0, 1].conjugate()).real
                  - 2 * C * (fa * F[0, 1].conjugate() + F[0, 0] * fb.conjugate()).real)
            grad[i, j] = 2 * (dN * D - N * (dA * B + A * dB - 2 * C * dC)) / (D * D)
    return two_f, grad


def exact(case, seed):
    c = case
    if c["kind"] == "dense":
        bank = _bank(_rng(seed), c)
        return torch.stack(list(_exact_rows(c, *_series(c, seed, bank), bank)))
    if c["kind"] == "peaks":
        bank = _bank(_rng(seed), c)
        rows = _exact_rows(c, *_series(c, seed, bank), bank)
        best = torch.stack([r.reshape(c["bands"], -1).amax(1) for r in rows])
        return {"count": None, "band_max": best, "band_bin": None, "tmpl": None, "bin": None, "twoF": None}
    if c["kind"] == "batch":
        outs = []
        for k, t in enumerate(_targets(c)):
            bank = _bank(_rng(seed, 100 + k), t)
            outs.append(torch.stack(list(_exact_rows(t, *_series(t, seed, bank, sub=k), bank))))
        return outs
    if c["kind"] == "semi":
        bank, t_ref, parts = _segments(c, seed)
        n_fft, df = c["n_fft"], 1.0 / (c["n_fft"] * c["dt"])
        total = torch.zeros((len(bank), n_fft), dtype=torch.float64, device="cuda")
        for t0, xs, sigmas in parts:
            D = t0 + (c["n"] // 2) * c["dt"] - t_ref
            moved = bank.copy()
            moved["f1dot"] += bank["f2dot"] * D
            for i, r in enumerate(_exact_rows(c, xs, sigmas, moved, t0)):
                k = int(np.rint((bank["f1dot"][i] * D + 0.5 * bank["f2dot"][i] * D * D) / df))
                lo, hi = max(0, -k), min(n_fft, n_fft - k)
                if hi > lo:
                    total[i, lo:hi] += r[lo + k:hi + k]
        return {"sum": total, "band_max": total.reshape(len(bank), c["bands"], -1).amax(2), "band_bin": None}
    if c["kind"] == "grad":
        bank, cand = _candidates(c, seed)
        two_f, g = _exact_grad(c, *_series(c, seed, bank), cand)
        return {"twoF": two_f, "grad": g}
    if c["kind"] == "sft":
        full, bank, bins, m_raw = _sfts(c, seed)
        B = c["n_bins"]
        m = torch.arange(B, device="cuda", dtype=torch.float64)
        t_s = torch.arange(c["n_sft"], device="cuda", dtype=torch.float64) * c["t_sft"]
        turn = _turns(-((B // 2) * m % B) / B)[None, :] * _turns(-full["f_het"] * t_s)[:, None]
        xs = [(torch.fft.ifft(b.to(torch.complex128), dim=1) * (B / m_raw) * turn).reshape(-1) for b in bins]
        return torch.stack(list(_exact_rows(full, xs, [1.0] * c["det"], bank)))
    pairs, abc, tau0, f1dot, f2dot = _resampled(c, seed)
    g = torch.view_as_complex(pairs.double().reshape(-1, 2, 2).contiguous())
    tau = tau0 + torch.arange(c["n"], dtype=torch.float64, device="cuda") * c["dt"]
    return _exact_row(g[:, 0], g[:, 1], abc, tau, f1dot, f2dot, c["n_fft"])
