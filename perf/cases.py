"""The work a user of this library has it do, as cases that can be timed.

A case names one public entry point, a footprint, the catalogue sizes and a
bin range.  Sizes, footprints and bins are those of the repository's own
workloads (paper_1208_3658_gb300/synth.py) and tests, from the smallest
served request to the full-sky catalogue; points are drawn on the GPU.

  listed()            the named cases
  draw(rng)           one more case of the same ranges
  prepare(case, seed) inputs, plans and handles a program has before the call
  run(state)          one pass through the public entry point
  work(case)          bytes and operations one pass cannot do without
  exact(case, seed)   the same outputs in plain FP64, where that is quick
"""
import math

import numpy as np
import torch

from paper_1208_3658_gb300 import wtheta as W

DEG = math.pi / 180.0
ARCMIN = 1.0 / 60.0

# footprints: RA/Dec patches [ra0, ra1) x [dec0, dec1), a polar cap, the sky
PATCHES = {"patch10": (0.0, 10.0, 0.0, 10.0), "patch15": (120.0, 135.0, 20.0, 35.0)}
CAP_DEG = 60.0

# bin ranges: (lowest edge, highest edge, bins, mode)
BINS = {
    "small": (1.0 * ARCMIN, 5.0, 16, "log"),
    "serve": (1.0 * ARCMIN, 10.0, 24, "log"),
    "survey": (0.5 * ARCMIN, 20.0, 32, "log"),
    "largest": (0.2 * ARCMIN, 30.0, 64, "log"),
    "fine": (0.5 * ARCMIN, 20.0, 256, "log"),
    "linear": (0.0, 180.0, 36, "linear"),
}


def listed():
    return [
        # the smallest request that the server workload draws: launches and latency
        {"name": "wtheta_1k", "call": "wtheta", "foot": "patch15", "bins": "serve",
         "n_d": 1000, "n_r": 1000},
        # the small workload end to end: host RA/Dec in, counts and w(theta) out
        {"name": "correlate_10k", "call": "correlate", "foot": "patch10", "bins": "small",
         "n_d": 10000, "n_r": 10000},
        # one cross count of unit vectors that the caller already holds, ragged sizes
        {"name": "cross_xyz_30k_48k", "call": "cross_xyz", "foot": "patch15", "bins": "serve",
         "n_d": 30011, "n_r": 47777},
        # the entry that never allocates (no sort, no culling), ragged size
        {"name": "noalloc_20k", "call": "noalloc", "foot": "patch10", "bins": "small",
         "n_d": 20001, "n_r": 20001},
        # ordinary: a survey sample with three times as many randoms
        {"name": "wtheta_100k_300k", "call": "wtheta", "foot": "cap", "bins": "survey",
         "n_d": 100003, "n_r": 300007},
        # the paper's linear bins over the whole range: nothing is out of range
        {"name": "linear_sky_100k", "call": "wtheta", "foot": "sky", "bins": "linear",
         "n_d": 100000, "n_r": 100000},
        # the largest bin count the library takes
        {"name": "fine_bins_200k", "call": "wtheta", "foot": "cap", "bins": "fine",
         "n_d": 200000, "n_r": 200000},
        # jackknife: region-pair counts of 64 regions
        {"name": "regions_300k", "call": "regions", "foot": "cap", "bins": "survey",
         "n_d": 300000, "n_r": 300000, "regions": 64},
        # mock catalogues of uneven sizes through one kept batch plan
        {"name": "batch_16", "call": "batch", "foot": "patch15", "bins": "small",
         "mocks": 16, "n_lo": 20000, "n_hi": 400000},
        # a burst of requests to a running server, 70% auto and 30% cross
        {"name": "serve_24", "call": "serve", "foot": "patch15", "bins": "serve",
         "requests": 24, "n_lo": 1000, "n_hi": 200000},
        # the survey workload: the benchmark's step
        {"name": "survey_1m", "call": "wtheta", "foot": "cap", "bins": "survey",
         "n_d": 1000000, "n_r": 1000000},
        # a full-sky catalogue of the largest workload's shape
        {"name": "sky_5m", "call": "wtheta", "foot": "sky", "bins": "largest",
         "n_d": 5000000, "n_r": 5000000},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    call = rng.choice(["wtheta", "wtheta", "wtheta", "correlate", "cross_xyz", "noalloc",
                       "regions", "batch", "serve"])
    if call == "noalloc":
        n = _log_int(rng, 1000, 120000)
        return {"call": call, "foot": rng.choice(["patch10", "cap"]), "bins": "small",
                "n_d": n, "n_r": n}
    if call == "regions":
        n = _log_int(rng, 20000, 500000)
        return {"call": call, "foot": "cap", "bins": "survey", "n_d": n,
                "n_r": _log_int(rng, n, 2 * n), "regions": rng.randint(4, 100)}
    if call == "batch":
        return {"call": call, "foot": "patch15", "bins": "small", "mocks": rng.randint(2, 20),
                "n_lo": _log_int(rng, 2000, 20000), "n_hi": _log_int(rng, 40000, 400000)}
    if call == "serve":
        return {"call": call, "foot": "patch15", "bins": "serve", "requests": rng.randint(4, 30),
                "n_lo": _log_int(rng, 1000, 5000), "n_hi": _log_int(rng, 20000, 200000)}
    foot = rng.choice(["patch10", "patch15", "cap", "sky"])
    bins = {"patch10": ["small"], "patch15": ["serve", "small"], "cap": ["survey", "fine"],
            "sky": ["largest", "linear"]}[foot]
    bins = rng.choice(bins)
    hi = {"patch10": 400000, "patch15": 400000, "cap": 1000000, "sky": 2000000}[foot]
    if bins == "linear":
        hi = 300000
    if call == "correlate":
        hi = min(hi, 200000)
    n = _log_int(rng, 1000, hi)
    return {"call": call, "foot": foot, "bins": bins, "n_d": n, "n_r": _log_int(rng, n, 2 * n)}


# --------------------------------------------------------------------------
# inputs
# --------------------------------------------------------------------------
def _edges(case):
    lo, hi, k, mode = BINS[case["bins"]]
    return W.wtheta_edges(lo, hi, k, W.BINS_LINEAR if mode == "linear" else W.BINS_LN)


def _uniform(foot, n, g):
    u = torch.rand(2, n, generator=g, device="cuda", dtype=torch.float64)
    if foot in PATCHES:
        ra0, ra1, d0, d1 = PATCHES[foot]
        ra = ra0 + (ra1 - ra0) * u[0]
        z = math.sin(d0 * DEG) + (math.sin(d1 * DEG) - math.sin(d0 * DEG)) * u[1]
    else:
        ra = 360.0 * u[0]
        z0 = math.cos(CAP_DEG * DEG) if foot == "cap" else -1.0
        z = z0 + (1.0 - z0) * u[1]
    return torch.stack([ra, torch.asin(z.clamp(-1.0, 1.0)) / DEG], dim=1)


def _inside(foot, p):
    if foot in PATCHES:
        ra0, ra1, d0, d1 = PATCHES[foot]
        return (p[:, 0] >= ra0) & (p[:, 0] < ra1) & (p[:, 1] >= d0) & (p[:, 1] < d1)
    if foot == "cap":
        return p[:, 1] >= 90.0 - CAP_DEG
    return torch.ones(p.shape[0], dtype=torch.bool, device=p.device)


def _clustered(foot, n, g):
    """n points around n / 50 uniform centres (about 50 members each), Gaussian
    offsets in the tangent plane, members outside the footprint left out."""
    sigma = {"cap": 2.0, "sky": 1.0}.get(foot, 3.0) * ARCMIN * DEG
    got, have, per = [], 0, max(1, math.ceil(n / 50))
    while have < n:
        c = _uniform(foot, per, g) * DEG
        m = per * 52
        i = torch.randint(per, (m,), generator=g, device="cuda")
        ra, dec = c[i, 0], c[i, 1]
        off = sigma * torch.randn(2, m, generator=g, device="cuda", dtype=torch.float64)
        ca, sa, cd, sd = ra.cos(), ra.sin(), dec.cos(), dec.sin()
        x = cd * ca - off[0] * sa - off[1] * sd * ca
        y = cd * sa + off[0] * ca - off[1] * sd * sa
        z = sd + off[1] * cd
        p = torch.stack([torch.remainder(torch.atan2(y, x) / DEG, 360.0),
                         torch.atan2(z, torch.hypot(x, y)) / DEG], dim=1)
        p = p[_inside(foot, p)]
        got.append(p)
        have += p.shape[0]
    return torch.cat(got)[:n].contiguous()


def _xyz(rd):
    """Unit vectors (3, n) of RA/Dec (n, 2), as a user's own code makes them."""
    a, d = rd[:, 0] * DEG, rd[:, 1] * DEG
    return torch.stack([d.cos() * a.cos(), d.cos() * a.sin(), d.sin()]).contiguous()


def _sizes(case, count, stream):
    """Uneven sizes, log-uniform in [n_lo, n_hi], the same for every seed (they
    are the case's, not the inputs')."""
    u = np.random.default_rng([case["n_lo"], case["n_hi"], count, stream]).random(count)
    lo, hi = math.log(case["n_lo"]), math.log(case["n_hi"])
    return [int(round(math.exp(lo + (hi - lo) * v))) for v in u]


def _is_cross(q):
    return q % 10 in (2, 5, 8)  # 30% of a stream of requests


def prepare(case, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    e, call, foot = _edges(case), case["call"], case["foot"]
    s = {"call": call, "edges": e}
    if call == "batch":
        s["cats"] = [(_clustered(foot, n, g), _uniform(foot, 2 * n, g))
                     for n in _sizes(case, case["mocks"], 1)]
        s["plan"] = W.wtheta_batch_plan(s["cats"], e)
        s["counts"] = torch.empty(case["mocks"] * 3 * (len(e) + 1), dtype=torch.int64,
                                  device="cuda")
        return s
    if call == "serve":
        host = lambda t: t.cpu().numpy().reshape(-1)  # noqa: E731
        s["requests"] = []
        for q, n in enumerate(_sizes(case, case["requests"], 2)):
            r = [host(_clustered(foot, n, g)), host(_uniform(foot, n, g))]
            if _is_cross(q):
                r += [host(_clustered(foot, n, g)), host(_uniform(foot, n, g))]
            s["requests"].append(r)
        s["server"] = W.wtheta_server_create(e, 8 << 30)
        return s
    d, r = _clustered(foot, case["n_d"], g), _uniform(foot, case["n_r"], g)
    if call == "correlate":
        s["d"], s["r"] = d.cpu().numpy().reshape(-1), r.cpu().numpy().reshape(-1)
        return s
    n_counts = 3
    if call in ("cross_xyz", "noalloc"):
        d, r, n_counts = _xyz(d), _xyz(r), 1
    if call == "regions":
        R = n_counts = case["regions"]
        n_counts *= 3 * R
        # regions: equal steps of RA
        s["labels"] = [(p[:, 0] / 360.0 * R).floor().clamp(0, R - 1).to(torch.int32)
                       for p in (d, r)]
        s["regions"] = R
    s["d"], s["r"] = d, r
    s["counts"] = torch.empty(n_counts * (len(e) + 1), dtype=torch.int64, device="cuda")
    return s


# --------------------------------------------------------------------------
# one pass
# --------------------------------------------------------------------------
def run(s):
    call, e = s["call"], s["edges"]
    if call == "correlate":
        counts, w = W.wtheta_correlate(s["d"], s["r"], e)
        return {"counts": counts.view(np.int64), "w": w}
    if call == "wtheta":
        W.wtheta_count_wtheta(s["d"], s["r"], False, e, s["counts"])
    elif call == "cross_xyz":
        W.wtheta_count_xyz(s["d"], s["r"], e, False, s["counts"])
    elif call == "noalloc":
        W.wtheta_count_xyz_noalloc(s["d"], None, e, True, s["counts"])
    elif call == "regions":
        sizes = W.wtheta_count_regions(s["d"], s["labels"][0], s["r"], s["labels"][1], e,
                                       s["regions"], s["counts"])
        return {"counts": s["counts"], "sizes": sizes}
    elif call == "batch":
        W.wtheta_batch_run(s["plan"], s["counts"])
    elif call == "serve":
        srv = s["server"]
        ids = [W.wtheta_server_submit(srv, *q) for q in s["requests"]]
        counts, w = [], []
        for i in ids:
            _, c, x = W.wtheta_server_wait(srv, i)
            W.wtheta_server_release(srv, i)
            counts.append(c.reshape(-1))
            w.append(x)
        return {"counts": np.concatenate(counts).view(np.int64), "w": np.stack(w)}
    return {"counts": s["counts"]}


# --------------------------------------------------------------------------
# what a pass cannot do without
# --------------------------------------------------------------------------
def _in_range(case):
    """About the fraction of the pairs that lie below the top edge: only those
    have to be told apart (6 operations per squared chord)."""
    theta = BINS[case["bins"]][1] * DEG
    cap = 0.5 * (1.0 - math.cos(theta))
    if case["foot"] in PATCHES:
        ra0, ra1, d0, d1 = PATCHES[case["foot"]]
        sky = (ra1 - ra0) * DEG * (math.sin(d1 * DEG) - math.sin(d0 * DEG)) / (4.0 * math.pi)
    else:
        sky = 0.5 * (1.0 - math.cos(CAP_DEG * DEG)) if case["foot"] == "cap" else 1.0
    return min(1.0, cap / sky)


def work(case):
    slots = BINS[case["bins"]][2] + 2
    auto = lambda n: n * (n - 1) / 2.0  # noqa: E731
    call = case["call"]
    if call == "batch":
        n = _sizes(case, case["mocks"], 1)
        pairs = sum(auto(k) + 2.0 * k * k + auto(2 * k) for k in n)
        nbytes = sum(16 * 3 * k + 8 * 3 * slots for k in n)
    elif call == "serve":
        pairs = nbytes = 0
        for q, k in enumerate(_sizes(case, case["requests"], 2)):
            pairs += 4.0 * k * k if _is_cross(q) else 2 * auto(k) + 1.0 * k * k
            nbytes += 16 * k * (4 if _is_cross(q) else 2) + 8 * slots * (4 if _is_cross(q) else 3)
    elif call == "noalloc":
        pairs, nbytes = auto(case["n_d"]), 24 * case["n_d"] + 8 * slots
    elif call == "cross_xyz":
        pairs = 1.0 * case["n_d"] * case["n_r"]
        nbytes = 24 * (case["n_d"] + case["n_r"]) + 8 * slots
    else:
        n_d, n_r = case["n_d"], case["n_r"]
        pairs = auto(n_d) + 1.0 * n_d * n_r + auto(n_r)
        nbytes = 16 * (n_d + n_r) + 24 * slots
        if call == "regions":
            nbytes += 4 * (n_d + n_r) + 24 * slots * (case["regions"] ** 2 - 1)
    return {"bytes": nbytes, "flops": 6.0 * pairs * _in_range(case)}


# --------------------------------------------------------------------------
# the same in plain FP64
# --------------------------------------------------------------------------
def _count_fp64(a, b, c, auto):
    """Pairs per slot of the squared chord |a - b|^2 against the edges c."""
    out = torch.zeros(len(c) + 1, dtype=torch.int64, device="cuda")
    rows = max(1, (1 << 26) // b.shape[1])
    j = torch.arange(b.shape[1], device="cuda")
    for i0 in range(0, a.shape[1], rows):
        p = a[:, i0:i0 + rows]
        q = [p[k][:, None] - b[k][None, :] for k in range(3)]
        t = (q[0] * q[0] + q[1] * q[1]) + q[2] * q[2]
        if auto:
            t = t[torch.arange(i0, i0 + p.shape[1], device="cuda")[:, None] < j[None, :]]
        slot = torch.bucketize(t.reshape(-1), c, right=True)
        out += torch.bincount(slot, minlength=len(c) + 1)
    return out


def exact(case, seed):
    if case["call"] != "correlate" or max(case["n_d"], case["n_r"]) > 60000:
        return None
    s = prepare(case, seed)
    d, r = (_xyz(torch.from_numpy(s[k]).reshape(-1, 2).cuda()) for k in ("d", "r"))
    edges = torch.from_numpy(s["edges"]).cuda()
    c = 4.0 * torch.sin(edges * (math.pi / 360.0)) ** 2
    n = [_count_fp64(d, d, c, True), _count_fp64(d, r, c, False), _count_fp64(r, r, c, True)]
    dd, dr, rr = (v[1:-1].double() / v.sum().double() for v in n)
    return {"counts": None, "w": ((dd - 2.0 * dr + rr) / rr).cpu().numpy()}
