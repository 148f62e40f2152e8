"""Timed cases of the k-NN query path, through the public entry points.

Every case is what a program does over and over with a cloud it has built and
uploaded once: queries from anywhere in a padded box around a sampled surface
("volume"), just off the surface ("surface"), half of each ("mixed"), the
cloud's own sites, many clouds in one captured plan, requests through the
server, queries and results in host memory. Surfaces, orders and query
distributions are those of the synthetic workloads (random insertion order;
box padded by 0.2; |N(0, 0.01)| off the surface; m log-uniform in [1000, n];
requests of 1..65,536 queries, k in 1..64, m in [n/10, n]).

A cloud is built once per process and shared by the states of every seed, as
a program keeps it; queries, bounds and requests come from the seed.
"""
from __future__ import annotations

import math
from concurrent.futures import ThreadPoolExecutor

import torch

from paper_2605_02224_gb300 import Cloud
from paper_2605_02224_gb300 import mknn as M

_SURFACES = ("sphere", "torus", "bumpy", "patches")
_PAD = 0.2
# pairs (query, site) that a brute-force answer in 64 bits may take
_EXACT_PAIRS = 1.05e11


def listed():
    return [
        # one small lookup in a small cloud (interactive picking, a simulation's
        # probe points): launch latency and the longest single query
        {"name": "small_call", "do": "query", "surface": "sphere", "n": 2000, "nq": 64,
         "queries": "volume", "k": 8, "m": 0},
        # an ordinary call of a loop over frames or scans
        {"name": "scan_10k", "do": "query", "surface": "torus", "n": 100_000, "nq": 10_007,
         "queries": "mixed", "k": 8, "m": 0},
        # the headline: a large batch of volume queries on a 1M-point surface
        {"name": "volume_4m_k16", "do": "query", "surface": "torus", "n": 1_000_000,
         "nq": 4_000_000, "queries": "volume", "k": 16, "m": 0},
        # distance fields and projections: few neighbours, many points
        {"name": "field_1m_k4", "do": "query", "surface": "bumpy", "n": 300_000,
         "nq": 999_983, "queries": "volume", "k": 4, "m": 0},
        # neighbourhoods for local fits
        {"name": "fit_500k_k32", "do": "query", "surface": "torus", "n": 1_000_000,
         "nq": 500_000, "queries": "mixed", "k": 32, "m": 0},
        # wide neighbourhoods (outlier statistics, descriptors)
        {"name": "wide_100k_k100", "do": "query", "surface": "torus", "n": 1_000_000,
         "nq": 100_000, "queries": "surface", "k": 100, "m": 0},
        # level of detail: every query sees its own prefix of the cloud
        {"name": "prefix_1m5_k10", "do": "query", "surface": "bumpy", "n": 300_000,
         "nq": 1_500_000, "queries": "mixed", "k": 10, "m": "each"},
        # the cloud against itself (normals, smoothing): every site a query
        {"name": "sites_1m_k16", "do": "sites", "surface": "torus", "n": 1_000_000,
         "nq": 1_000_000, "k": 16, "m": 0},
        # near-planar scans: a few sites with very long successor lists
        {"name": "planar_200k_k8", "do": "query", "surface": "patches", "n": 200_000,
         "nq": 200_001, "queries": "mixed", "k": 8, "m": 0},
        # many clouds in one captured plan, two queries per point
        {"name": "plan_12", "do": "plan", "clouds": 12, "lo": 10_000, "hi": 80_000, "mix": 21},
        # a burst of requests through the server, host buffers in and out
        {"name": "serve_64", "do": "serve", "clouds": 4, "lo": 50_000, "hi": 200_000, "mix": 41,
         "requests": 64, "max_q": 65_536},
        # queries and results in (pinned) host memory
        {"name": "host_2m_k8", "do": "host", "surface": "torus", "n": 1_000_000,
         "nq": 2_000_000, "queries": "volume", "k": 8, "m": 0},
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(math.exp(rng.uniform(math.log(lo), math.log(hi))))))


def draw(rng):
    do = rng.choice(["query"] * 6 + ["sites", "plan", "serve", "host"])
    if do == "plan":
        return {"do": "plan", "clouds": rng.randint(3, 16), "lo": rng.randint(4000, 10_000),
                "hi": rng.randint(20_000, 60_000), "mix": rng.randint(100, 1 << 20)}
    if do == "serve":
        return {"do": "serve", "clouds": rng.randint(2, 5), "lo": rng.randint(10_000, 50_000),
                "hi": rng.randint(60_000, 200_000), "mix": rng.randint(100, 1 << 20),
                "requests": rng.randint(8, 64), "max_q": _log_int(rng, 512, 65_536)}
    surface = rng.choice(_SURFACES)
    n = _log_int(rng, 2000, 400_000)
    k = _log_int(rng, 1, 128)
    # queries that take no longer than the largest listed case (about 9 ms)
    per_query_ns = (0.7 + 0.09 * k + 0.0022 * k * k) * (4 if surface == "patches" else 1)
    most = max(1000, min(2_000_000, int(6e6 / per_query_ns)))
    nq = _log_int(rng, 1, most)
    c = {"do": do, "surface": surface, "n": n, "nq": nq, "k": k,
         "m": rng.choice([0, 0, 0, "each", rng.randint(max(1, n // 10), n)])}
    if do != "sites":
        c["queries"] = rng.choice(["volume", "mixed", "surface"])
    return c


# ------------------------------------------------------------------- surfaces

def _gen(device, seed):
    return torch.Generator(device=device).manual_seed(int(seed))


def _unit(v):
    return v / v.norm(dim=-1, keepdim=True)


def _surface(kind, n, g):
    """n points of a surface and their unit normals, float64 on g's device."""
    dev = g.device
    two_pi = 2 * math.pi

    def rand(*s):
        return torch.rand(*s, generator=g, device=dev, dtype=torch.float64)

    def randn(*s):
        return torch.randn(*s, generator=g, device=dev, dtype=torch.float64)

    if kind == "sphere":
        d = _unit(randn(n, 3))
        return d, d
    if kind == "torus":  # R = 1, r = 0.3, uniform by area, N(0, 1e-4) along the normal
        th, have = [], 0
        while have < n:
            t = two_pi * rand(int(1.5 * n) + 64)
            t = t[rand(t.shape[0]) * 1.3 < 1.0 + 0.3 * torch.cos(t)]
            th.append(t)
            have += t.shape[0]
        th, ph = torch.cat(th)[:n], two_pi * rand(n)
        ct, st, cp, sp = torch.cos(th), torch.sin(th), torch.cos(ph), torch.sin(ph)
        nrm = torch.stack([ct * cp, ct * sp, st], 1)
        p = torch.stack([(1.0 + 0.3 * ct) * cp, (1.0 + 0.3 * ct) * sp, 0.3 * st], 1)
        return p + 1e-4 * randn(n, 1) * nrm, nrm
    if kind == "bumpy":  # radius 1 + 0.1 sin(8 theta) sin(8 phi) over uniform directions
        d = _unit(randn(n, 3))
        th = torch.arccos(d[:, 2].clamp(-1.0, 1.0))
        ph = torch.arctan2(d[:, 1], d[:, 0])
        st, ct, sp, cp = torch.sin(th), torch.cos(th), torch.sin(ph), torch.cos(ph)
        rho = 1.0 + 0.1 * torch.sin(8 * th) * torch.sin(8 * ph)
        r_th = 0.8 * torch.cos(8 * th) * torch.sin(8 * ph)
        r_ph = 0.8 * torch.sin(8 * th) * torch.cos(8 * ph)
        e_th = torch.stack([ct * cp, ct * sp, -st], 1)
        e_ph = torch.stack([-sp, cp, torch.zeros_like(ph)], 1)
        nrm = d - (r_th / rho)[:, None] * e_th - (r_ph / (rho * st.clamp(min=1e-12)))[:, None] * e_ph
        return rho[:, None] * d, _unit(nrm)
    # four planar squares of side 0.5 in the unit cube, the same ones for points and queries
    f = _gen("cpu", 7)
    ctr = 0.25 + 0.5 * torch.rand(4, 3, generator=f, dtype=torch.float64)
    nv = _unit(torch.randn(4, 3, generator=f, dtype=torch.float64))
    u = _unit(torch.linalg.cross(nv, torch.eye(3, dtype=torch.float64)[nv.abs().argmin(1)]))
    v = torch.linalg.cross(nv, u)
    ctr, nv, u, v = (t.to(dev) for t in (ctr, nv, u, v))
    i = torch.arange(n, device=dev) % 4
    st = 0.5 * (rand(n, 2) - 0.5)
    return ctr[i] + st[:, :1] * u[i] + st[:, 1:] * v[i], nv[i]


# --------------------------------------------------------------------- clouds

_points_of = {}  # (surface, n) -> its points on the host (input order), its insertion order
_clouds = {}     # (surface, n) -> Cloud


def _points(spec):
    if spec not in _points_of:
        kind, n = spec
        g = _gen("cpu", 1000 + n + _SURFACES.index(kind))
        points = _surface(kind, n, g)[0].float()
        _points_of[spec] = points, torch.randperm(n, generator=g)
    return _points_of[spec]


def _build(spec):
    points, order = _points(spec)
    return Cloud.build(points.numpy(), order.numpy())


def _get_clouds(specs):
    """The clouds of `specs`, the missing ones built at the same time."""
    missing = sorted({s for s in specs if s not in _clouds})
    with ThreadPoolExecutor(8) as pool:
        for s, c in zip(missing, pool.map(_build, missing)):
            _clouds[s] = c.upload()
    return [_clouds[s] for s in specs]


def _mix(case):
    """(surface, n, k) of each cloud of a plan or server: sizes log-uniform in [lo, hi]."""
    g = _gen("cpu", case["mix"])
    u = torch.rand(case["clouds"], 3, generator=g, dtype=torch.float64).tolist()
    lo, hi = math.log(case["lo"]), math.log(case["hi"])
    return [(_SURFACES[int(4 * a)], int(math.exp(lo + b * (hi - lo))), (1, 4, 8, 16, 32)[int(5 * c)])
            for a, b, c in u]


# -------------------------------------------------------------------- queries

def _queries(kind, points, how, nq, g):
    """(nq, 3) float32 on g's device."""
    lo = points.min(0).values.double().to(g.device) - _PAD
    hi = points.max(0).values.double().to(g.device) + _PAD
    nv = {"volume": nq, "surface": 0, "mixed": nq // 2}[how]
    box = lo + (hi - lo) * torch.rand(nv, 3, generator=g, device=g.device, dtype=torch.float64)
    if nv == nq:
        return box.float()
    p, nrm = _surface(kind, nq - nv, g)
    off = 0.01 * torch.randn(nq - nv, 1, generator=g, device=g.device, dtype=torch.float64).abs()
    return torch.cat([box, p + off * nrm]).float()


def _bounds(m, n, nq, g):
    """None, a number, or one bound per query (log-uniform in [min(1000, n), n])."""
    if m != "each":
        return m or None
    lo = math.log(min(1000, n))
    u = torch.rand(nq, generator=g, device=g.device, dtype=torch.float64)
    return torch.exp(lo + u * (math.log(n) - lo)).floor().clamp(1, n).to(torch.int32)


class _Plan:
    """A captured plan and its output rows; freed with the state."""

    def __init__(self, reqs):
        self.reqs = reqs
        self.handle = M.mknn_batch_create(reqs)

    def __del__(self):
        M.mknn_batch_free(self.handle)


_servers = {}  # the clouds of a server -> its handle, kept as a serving program keeps it


def _server(specs, clouds):
    key = tuple(specs)
    if key not in _servers:
        h = M.mknn_server_create(mem_budget=1 << 28)
        for c in clouds:
            M.mknn_server_add_cloud(h, c.handle)
        _servers[key] = h
    return _servers[key]


def _requests(case, seed):
    """The burst's requests: (cloud number, queries on the host, k, m). Who asks
    what (cloud, number of queries, k) belongs to the case, the queries and
    bounds to the seed."""
    mix = _mix(case)
    u = torch.rand(case["requests"], 3, generator=_gen("cpu", case["mix"] + 1),
                   dtype=torch.float64).tolist()
    g = _gen("cpu", seed)
    out = []
    for a, b, c in u:
        i = int(a * len(mix))
        kind, n, _ = mix[i]
        nq = max(1, min(case["max_q"], int(math.exp(b * math.log(case["max_q"])))))
        low = max(1, -(-n // 10))
        m = low + int(float(torch.rand(1, generator=g)) * (n - low + 1))
        out.append((i, _queries(kind, _points((kind, n))[0], "mixed", nq, g), 1 + int(64 * c),
                    min(n, m)))
    return out


# ---------------------------------------------------------------------- cases

def prepare(case, seed):
    do = case["do"]
    if do == "plan":
        mix = _mix(case)
        g = _gen("cuda", seed)
        reqs = []
        for (kind, n, k), cloud in zip(mix, _get_clouds([s[:2] for s in mix])):
            q = _queries(kind, _points((kind, n))[0], "mixed", 2 * n, g)
            reqs.append({"cloud": cloud.handle, "q": q, "nq": 2 * n, "q_stride": 3, "k": k,
                         "out_idx": torch.empty(2 * n, k, dtype=torch.int32, device="cuda"),
                         "out_d2": torch.empty(2 * n, k, dtype=torch.float32, device="cuda")})
        return {"do": do, "plan": _Plan(reqs)}
    if do == "serve":
        mix = _mix(case)
        specs = [s[:2] for s in mix]
        server = _server(specs, _get_clouds(specs))
        reqs = _requests(case, seed)
        q = torch.cat([r[1] for r in reqs]).pin_memory()
        rows = sum(r[1].shape[0] * r[2] for r in reqs)
        idx = torch.empty(rows, dtype=torch.int32, pin_memory=True)
        d2 = torch.empty(rows, dtype=torch.float32, pin_memory=True)
        calls, a, b = [], 0, 0
        for i, rq, k, m in reqs:
            nq = rq.shape[0]
            calls.append((i, q[a:a + nq], k, m, idx[b:b + nq * k], d2[b:b + nq * k]))
            a, b = a + nq, b + nq * k
        return {"do": do, "server": server, "calls": calls, "idx": idx, "d2": d2}
    n, nq, k = case["n"], case["nq"], case["k"]
    spec = (case["surface"], n)
    cloud = _get_clouds([spec])[0]
    points = _points(spec)[0]
    g = _gen("cuda", seed)
    if do == "sites":
        sites = torch.randperm(n, generator=g, device="cuda").to(torch.int32)
        sites = sites.repeat(-(-nq // n))[:nq].contiguous()
        return {"do": do, "cloud": cloud, "sites": sites, "k": k, "m": _bounds(case["m"], n, nq, g)}
    q = _queries(case["surface"], points, case["queries"], nq, g)
    m = _bounds(case["m"], n, nq, g)
    if do == "host":
        return {"do": do, "cloud": cloud, "q": q.cpu().pin_memory(), "k": k,
                "m": m.cpu().numpy() if torch.is_tensor(m) else m,
                "idx": torch.empty(nq, k, dtype=torch.int32, pin_memory=True),
                "d2": torch.empty(nq, k, dtype=torch.float32, pin_memory=True)}
    return {"do": do, "cloud": cloud, "q": q, "k": k, "m": m}


def run(state):
    do = state["do"]
    if do == "query":
        return state["cloud"].knn(state["q"], state["k"], state["m"])
    if do == "sites":
        return state["cloud"].knn_sites(state["sites"], state["k"], state["m"])
    if do == "host":
        return state["cloud"].knn_host(state["q"], state["k"], state["m"], state["idx"], state["d2"])
    if do == "plan":
        plan = state["plan"]
        M.mknn_batch_run(plan.handle, torch.cuda.current_stream().cuda_stream)
        return [(r["out_idx"], r["out_d2"]) for r in plan.reqs]
    for call in state["calls"]:
        M.mknn_server_submit(state["server"], *call)
    M.mknn_server_drain(state["server"])
    return state["idx"], state["d2"]


def _parts(case):
    """(sites, queries, k, queries carry a bound) of each cloud of a pass; for a
    burst of requests, the expected number and mean k."""
    if case["do"] == "plan":
        return [(n, 2 * n, k, False) for _, n, k in _mix(case)]
    if case["do"] == "serve":
        mean_q = case["max_q"] / max(1.0, math.log(case["max_q"]))
        per = max(1, int(case["requests"] * mean_q / case["clouds"]))
        return [(n, per, 32, False) for _, n, _ in _mix(case)]
    return [(case["n"], case["nq"], case["k"], case["m"] == "each")]


def work(case):
    """Coordinates of every site and query read once (a site query: its rank),
    bounds read once, rows written once; the k distances of each row."""
    bytes_, flops = 0, 0
    for n, nq, k, each in _parts(case):
        q = 4 if case["do"] == "sites" else 12
        bytes_ += 12 * n + nq * (q + (4 if each else 0) + 8 * k)
        flops += 8 * k * nq
    return {"bytes": bytes_, "flops": flops}


# -------------------------------------------------- 64-bit answers, brute force

def _brute(points, order, q, k, m):
    """The k smallest squared distances to the first m points in insertion
    order, ascending, +inf past m; float64."""
    p = points[order].double().cuda()
    n, nq = p.shape[0], q.shape[0]
    q = q.double().cuda()
    if torch.is_tensor(m):
        m = m.cuda().long()
    else:
        p = p[:m] if m else p
    out = torch.full((nq, k), math.inf, dtype=torch.float64, device="cuda")
    step = max(1, int(2.5e8) // p.shape[0])
    rank = torch.arange(p.shape[0], device="cuda")
    for a in range(0, nq, step):
        c = q[a:a + step]
        d = torch.zeros(c.shape[0], p.shape[0], dtype=torch.float64, device="cuda")
        for x in range(3):
            t = c[:, x:x + 1] - p[None, :, x]
            d.addcmul_(t, t)
        if torch.is_tensor(m):
            d.masked_fill_(rank[None, :] >= m[a:a + step, None], math.inf)
        kk = min(k, p.shape[0])
        out[a:a + step, :kk] = d.topk(kk, dim=1, largest=False).values.sort(dim=1).values
    return out


def exact(case, seed):
    """Distances only (ranks are whole numbers); None where brute force is too long."""
    if sum(n * nq for n, nq, _, _ in _parts(case)) > _EXACT_PAIRS:
        return None
    do = case["do"]
    if do == "plan":
        g = _gen("cuda", seed)
        out = []
        for kind, n, k in _mix(case):
            points, order = _points((kind, n))
            out.append((None, _brute(points, order, _queries(kind, points, "mixed", 2 * n, g), k, 0)))
        return out
    if do == "serve":
        specs = [s[:2] for s in _mix(case)]
        return None, torch.cat([_brute(*_points(specs[i]), q, k, m).reshape(-1)
                                for i, q, k, m in _requests(case, seed)])
    points, order = _points((case["surface"], case["n"]))
    n, nq, k = case["n"], case["nq"], case["k"]
    g = _gen("cuda", seed)
    if do == "sites":
        sites = torch.randperm(n, generator=g, device="cuda").repeat(-(-nq // n))[:nq]
        return None, _brute(points, order, points[order][sites.cpu()], k, _bounds(case["m"], n, nq, g))
    q = _queries(case["surface"], points, case["queries"], nq, g)
    return None, _brute(points, order, q, k, _bounds(case["m"], n, nq, g))
