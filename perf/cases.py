"""Workloads for timing the library through its public entry points.

A case is a dict of plain values. ``prepare`` makes what a program holds
before the call (a grid, its density, rays or points on the GPU or in pinned
host memory), ``run`` is one call as a program makes it, ``work`` the bytes
and operations of one call, ``exact`` its result in 64 bits by brute force
(every site a candidate, no neighbour lists) where that is affordable.

The shapes are those of ``bench.py``, ``gen/`` and the tests: uniform,
exponential-disk, clumpy and ball-shaped grids of 10^3 to 10^6 sites, 10^3
to 10^7 rays.
"""
import math

import numpy as np
import torch

from paper_1310_1854_gb300 import Batch, VoronoiGrid, optical_depth

CUBE = (-1.0, -1.0, -1.0, 1.0, 1.0, 1.0)
DISK = (-4.0, -4.0, -0.5, 4.0, 4.0, 0.5)
BALL = (0.0, 0.0, 0.0, 1.0)

# mean crossings per ray, in units of sites^(1/3) (measured on these shapes)
CROSSINGS = {"uniform": 0.7, "disk": 0.62, "clumpy": 0.64, "ball": 0.69, "detector": 2.0}
NEIGHBOURS = 15.5  # mean length of a neighbour list


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------

def listed():
    return [
        # a quick look at a small model: the whole call is latency
        {"name": "tau_small", "kind": "tau", "place": "uniform", "sites": 1000, "rays": 10_000,
         "precision": "fp32", "enter": False},
        # the benchmark: one Monte Carlo step's packages through a spiral-like disk
        {"name": "tau_disk", "kind": "tau", "place": "disk", "sites": 100_000, "rays": 1_000_000,
         "precision": "fp32", "enter": False},
        # the largest: a clumpy medium whose grid is beyond L2, many packages
        {"name": "tau_clumpy", "kind": "tau", "place": "clumpy", "sites": 1_000_000, "rays": 10_000_000,
         "precision": "fp32", "enter": False},
        # the same disk in float64, where the reference values come from
        {"name": "tau64_disk", "kind": "tau", "place": "disk", "sites": 100_000, "rays": 1_000_000,
         "precision": "fp64", "enter": False},
        # photons entering a spherical domain from outside, lengths exact to float32
        {"name": "tau_exact_ball", "kind": "tau", "place": "ball", "sites": 60_001, "rays": 300_007,
         "precision": "fp32_exact", "enter": True},
        # the paths themselves (cell and length lists), for a caller's own physics
        {"name": "segments_disk", "kind": "segments", "place": "disk", "sites": 100_000, "rays": 1_000_000,
         "precision": "fp32", "enter": False},
        # fitting densities to detector images: forward and backward
        {"name": "fit_disk", "kind": "fit", "place": "disk", "sites": 1_000_000, "rays": 1_000_000, "pixels": 512,
         "precision": "fp32", "keep": True},
        # Monte Carlo interaction points with the absorbed energy booked per cell
        {"name": "interact_disk", "kind": "interact", "place": "disk", "sites": 100_000, "rays": 1_000_000},
        # the cell of each of many points: grid-quality measure, sampling a model
        {"name": "locate_disk", "kind": "locate", "place": "disk", "sites": 1_000_000, "rays": 10_000_000,
         "precision": "fp32"},
        # a parameter study: many models of uneven size in one launch
        {"name": "batch16", "kind": "batch", "place": "mixed", "grids": 16, "sites": 200_000, "rays": 1_000_000},
        # packages produced on the host, optical depths wanted there
        {"name": "host_disk", "kind": "host", "place": "disk", "sites": 100_000, "rays": 1_000_000,
         "precision": "fp32"},
        # a new model: cells constructed, density set and a first set of rays traced
        {"name": "build_clumpy", "kind": "build", "place": "clumpy", "sites": 100_000, "rays": 100_000},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["tau", "tau", "tau", "segments", "segments", "fit", "interact", "locate", "batch", "host",
                       "build"])
    place = rng.choice(["uniform", "disk", "clumpy", "ball"])
    if kind == "batch":
        return {"kind": kind, "place": "mixed", "grids": rng.randint(2, 24), "sites": _log_int(rng, 4_000, 150_000),
                "rays": _log_int(rng, 20_000, 600_000)}
    if kind == "build":
        sites = _log_int(rng, 1_000, 100_000)
        return {"kind": kind, "place": place, "sites": sites, "rays": _log_int(rng, 1_000, 100_000)}
    sites = _log_int(rng, 1_000, 1_000_000)
    per_ray = CROSSINGS[place] * sites ** (1.0 / 3.0)
    precision = rng.choice(["fp32", "fp32", "fp64", "fp32_exact"])
    if kind == "locate":
        return {"kind": kind, "place": place, "sites": sites, "rays": _log_int(rng, 1_000, 10_000_000),
                "precision": rng.choice(["fp32", "fp32", "fp64"])}
    # crossings of the largest case of each kind
    most = {"tau": 6e8 if precision != "fp64" else 2.8e7, "segments": 2.8e7, "fit": 6e7, "interact": 2.8e7,
            "host": 2.8e7}[kind]
    rays = min(_log_int(rng, 1_000, 10_000_000), int(most / per_ray))
    if kind == "fit":
        return {"kind": kind, "place": place, "sites": sites, "rays": rays, "pixels": rng.randint(8, 200),
                "precision": rng.choice(["fp32", "fp32_exact"]), "keep": rng.random() < 0.5}
    if kind == "interact":
        return {"kind": kind, "place": place, "sites": sites, "rays": rays}
    case = {"kind": kind, "place": place, "sites": sites, "rays": rays, "precision": precision}
    if kind != "host":
        case["enter"] = rng.random() < 0.3
    return case


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _inside(p, box):
    return np.all((p >= np.array(box[:3])) & (p <= np.array(box[3:])), axis=1)


def _disk_draw(n, rng):
    R, phi, z = rng.gamma(2.0, 1.0, n), rng.uniform(0.0, 2.0 * math.pi, n), rng.laplace(0.0, 0.1, n)
    p = np.stack([R * np.cos(phi), R * np.sin(phi), z], axis=1)
    return p[_inside(p, DISK)]


def _distinct(p, n):
    """The first n distinct rows (float32 values as float64)."""
    b = np.ascontiguousarray(p).view(np.uint32).astype(np.uint64)
    key = (b[:, 0] * np.uint64(0x9E3779B97F4A7C15)) ^ (b[:, 1] * np.uint64(0xC2B2AE3D27D4EB4F)) ^ (
        b[:, 2] * np.uint64(0x165667B19E3779F9))
    first = np.sort(np.unique(key, return_index=True)[1])[:n]
    assert first.size == n
    return p[first].astype(np.float64)


def _model(place, n, seed):
    """(sites float64[n, 3] of float32 values, rho float32[n], box, sphere)."""
    rng = np.random.default_rng(seed)
    m = n + n // 50 + 64
    if place == "uniform":
        s = _distinct(rng.uniform(-1.0, 1.0, (m, 3)).astype(np.float32), n)
        return s, rng.uniform(0.5, 1.5, n).astype(np.float32), CUBE, None
    if place == "disk":
        p = np.concatenate([_disk_draw(m, rng) for _ in range(2)])
        s = _distinct(p.astype(np.float32), n)
        return s, np.exp(-np.hypot(s[:, 0], s[:, 1]) - np.abs(s[:, 2]) / 0.1).astype(np.float32), DISK, None
    if place == "ball":
        p = rng.uniform(-1.0, 1.0, (3 * m, 3)).astype(np.float32)
        s = _distinct(p[(p.astype(np.float64) ** 2).sum(axis=1) < 0.999999], n)
        return s, np.exp(-3.0 * np.linalg.norm(s, axis=1)).astype(np.float32), CUBE, BALL
    clumps = max(1, round(n / 500))
    centre = rng.uniform(-1.0, 1.0, (clumps, 3))
    sigma = np.exp(rng.uniform(math.log(0.01), math.log(0.05), clumps))
    which = rng.random(2 * m) < 0.3
    owner = rng.integers(0, clumps, 2 * m)
    p = np.where(which[:, None], centre[owner] + sigma[owner, None] * rng.standard_normal((2 * m, 3)),
                 rng.uniform(-1.0, 1.0, (2 * m, 3))).astype(np.float32)
    p, which = p[_inside(p, CUBE)], which[_inside(p, CUBE)]
    s = _distinct(p, n)
    b = np.ascontiguousarray(p[which]).view(np.uint32).astype(np.uint64)
    # dense where the site was drawn from a clump
    sb = np.ascontiguousarray(s.astype(np.float32)).view(np.uint32).astype(np.uint64)
    mix = lambda q: q[:, 0] << np.uint64(32) | (q[:, 1] ^ (q[:, 2] << np.uint64(7)))  # noqa: E731
    return s, np.where(np.isin(mix(sb), mix(b)), 100.0, 1.0).astype(np.float32), CUBE, None


def _points(place, n, seed):
    """Start points in the medium, drawn as its sites are (uniform for clumpy)."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    u = lambda k: torch.rand(k, 3, generator=g, device="cuda", dtype=torch.float64)  # noqa: E731
    if place == "disk":
        out = torch.empty(0, 3, device="cuda", dtype=torch.float64)
        while out.shape[0] < n:
            v = torch.rand(int(1.2 * n) + 64, 4, generator=g, device="cuda", dtype=torch.float64).clamp_min(1e-300)
            R = -torch.log(v[:, 0]) - torch.log(v[:, 1])
            phi = 2.0 * math.pi * v[:, 2]
            w = v[:, 3] - 0.5
            z = -0.1 * torch.sign(w) * torch.log1p((-2.0 * w.abs()).clamp_min(-1.0 + 1e-16))
            p = torch.stack([R * torch.cos(phi), R * torch.sin(phi), z], dim=1)
            keep = (p[:, :2].abs() <= 4.0).all(dim=1) & (z.abs() <= 0.5)
            out = torch.cat([out, p[keep]])
        return out[:n].contiguous()
    if place == "ball":
        out = torch.empty(0, 3, device="cuda", dtype=torch.float64)
        while out.shape[0] < n:
            p = 2.0 * u(2 * n + 64) - 1.0
            out = torch.cat([out, p[(p * p).sum(dim=1) < 0.9999]])
        return out[:n].contiguous()
    return 2.0 * u(n) - 1.0


def _directions(n, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    k = torch.randn(n, 3, generator=g, device="cuda", dtype=torch.float64)
    return k / torch.linalg.vector_norm(k, dim=1, keepdim=True).clamp_min(1e-12)


def _rays(place, n, seed, enter):
    p = _points(place, n, seed + 1)
    k = _directions(n, seed + 2)
    if enter:  # from outside: back along the ray, well out of the domain, still aimed at p
        p = (p - 12.0 * k).contiguous()
    return p, k


def _detector(npix, seed):
    """+x rays from the x = -4 (disk) or x = -1 face, one per pixel, jittered."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    j = torch.rand(npix * npix, 2, generator=g, device="cuda", dtype=torch.float64)
    i = torch.arange(npix * npix, device="cuda")
    return (torch.stack([i // npix, i % npix], dim=1) + j) / npix


def _same_length(case, seed):
    """Segment lists have as many entries as the scene has crossings, so every
    seed mirrors one scene in other axes, relabels its cells, gives them other
    densities and shoots its rays in another order: the lists keep their
    length and nothing else."""
    place, n, base = case["place"], case["rays"], case["sites"]
    sites, rho, box, sphere = _model(place, case["sites"], base)
    O, D = _rays(place, n, base, case.get("enter", False))
    rng = np.random.default_rng(seed)
    flip = rng.choice([-1.0, 1.0], 3)
    label = rng.permutation(case["sites"])
    rho = (rho[label] * np.exp(0.1 * rng.standard_normal(case["sites"]))).astype(np.float32)
    f = torch.from_numpy(flip).cuda()
    order = torch.randperm(n, generator=torch.Generator(device="cuda").manual_seed(seed), device="cuda")
    return {"sites": np.ascontiguousarray(sites[label] * flip), "rho": rho, "box": box, "sphere": sphere,
            "O": (O[order] * f).contiguous(), "D": (D[order] * f).contiguous()}


def _inputs(case, seed):
    """Everything that the call takes, without the grid object."""
    kind, place, n = case["kind"], case["place"], case["rays"]
    if kind == "segments":
        return _same_length(case, seed)
    sites, rho, box, sphere = _model(place, case["sites"], seed)
    d = {"sites": sites, "rho": rho, "box": box, "sphere": sphere}
    if kind == "locate":
        lo = torch.tensor(box[:3], device="cuda", dtype=torch.float64)
        hi = torch.tensor(box[3:], device="cuda", dtype=torch.float64)
        g = torch.Generator(device="cuda").manual_seed(seed + 1)
        d["O"] = lo + (hi - lo) * torch.rand(n, 3, generator=g, device="cuda", dtype=torch.float64)
        return d
    d["O"], d["D"] = _rays(place, n, seed, case.get("enter", False))
    g = torch.Generator(device="cuda").manual_seed(seed + 3)
    if kind == "interact":
        d["tau_int"] = -torch.log(torch.rand(n, generator=g, device="cuda").clamp_min(1e-30))
    if kind == "fit":
        npix = case["pixels"]
        yz = _detector(npix, seed + 4)
        lo, hi = (box[1], box[2]), (box[4], box[5])
        scale = 0.55 if sphere is not None else 1.0  # inside the ball's square cross-section
        y = scale * (lo[0] + (hi[0] - lo[0]) * yz[:, 0])
        z = scale * (lo[1] + (hi[1] - lo[1]) * yz[:, 1])
        x = -torch.sqrt(0.999 - y * y - z * z) if sphere is not None else torch.full_like(y, box[0])
        o = torch.stack([x, y, z], dim=1)
        k = torch.zeros_like(o)
        k[:, 0] = 1.0
        d["O"], d["D"] = torch.cat([o, d["O"]]).contiguous(), torch.cat([k, d["D"]]).contiguous()
        d["target"] = torch.rand(d["O"].shape[0], generator=g, device="cuda")
    return d


def _batch_plan(case):
    """Grid sizes and ray counts spread over their logarithm, the two kinds in turn."""
    rng = np.random.default_rng(case["sites"] + case["rays"])
    G = case["grids"]
    M = np.exp(rng.uniform(math.log(2_000), math.log(case["sites"]), G)).astype(int)
    N = np.exp(rng.uniform(math.log(10_000), math.log(case["rays"]), G)).astype(int)
    return [("uniform" if i % 2 == 0 else "disk", int(M[i]), int(N[i])) for i in range(G)]


def _grid(d):
    vg = VoronoiGrid(d["sites"], d["box"], sphere=d["sphere"], gpu_build=True)
    vg.set_density(torch.from_numpy(d["rho"]).cuda())
    return vg


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        sets = []
        for i, (place, M, N) in enumerate(_batch_plan(case)):
            s = seed + 1009 * (i + 1)
            sub = _inputs({"kind": "tau", "place": place, "sites": M, "rays": N}, s)
            sets.append((_grid(sub), sub["O"], sub["D"]))
        return {"case": case, "batch": Batch(sets)}
    d = _inputs(case, seed)
    st = {"case": case}
    for k in ("O", "D", "tau_int", "target"):
        if k in d:
            st[k] = d[k]
    if kind == "build":
        st.update(sites=d["sites"], box=d["box"], sphere=d["sphere"], rho=torch.from_numpy(d["rho"]).cuda())
        return st
    st["grid"] = _grid(d)
    if kind == "fit":
        st["rho"] = torch.from_numpy(d["rho"]).cuda()
    if kind == "host":
        st["O"], st["D"] = d["O"].cpu().pin_memory(), d["D"].cpu().pin_memory()
        dt = torch.float64 if case["precision"] == "fp64" else torch.float32
        st["out"] = torch.empty(case["rays"], dtype=dt, pin_memory=True)
    return st


# ---------------------------------------------------------------------------
# one call
# ---------------------------------------------------------------------------

def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "batch":
        state["batch"].run()
        return list(state["batch"].tau)
    if kind == "build":
        vg = VoronoiGrid(state["sites"], state["box"], sphere=state["sphere"], gpu_build=True)
        vg.set_density(state["rho"])
        volume, bbox = vg.cells()
        return [vg.trace(state["O"], state["D"]).tau, volume, bbox]
    vg = state["grid"]
    if kind == "tau":
        return vg.trace(state["O"], state["D"], precision=case["precision"], enter=case["enter"]).tau
    if kind == "segments":
        r = vg.trace(state["O"], state["D"], precision=case["precision"], segments=True, enter=case["enter"])
        return [r.tau, r.seg_len, r.seg_off, r.seg_cell]
    if kind == "locate":
        return vg.locate(state["O"], precision=case["precision"])
    if kind == "interact":
        cell, s, absorbed = vg.interact(state["O"], state["D"], state["tau_int"], absorbed=True)
        return [cell, s, absorbed]
    if kind == "host":
        return vg.trace_host(state["O"], state["D"], precision=case["precision"], out_tau=state["out"]).tau
    # fit: the loss of exp(-tau) against an image, and its gradient in the densities
    rho = state["rho"].detach().requires_grad_()
    tau = optical_depth(vg, rho, state["O"], state["D"], keep_segments=case["keep"], precision=case["precision"])
    loss = (torch.exp(-tau) - state["target"]).square().sum()
    loss.backward()
    return [tau.detach(), rho.grad]


# ---------------------------------------------------------------------------
# what one call cannot do without
# ---------------------------------------------------------------------------

def _trace_work(place, sites, rays, out_bytes):
    """Rays and the grid read once (site, list offset, neighbours, density),
    the outputs written; per crossing the planes of one cell."""
    x = rays * max(1.0, CROSSINGS[place] * sites ** (1.0 / 3.0))
    return {"bytes": 48.0 * rays + sites * (12.0 + 4.0 + 4.0 * NEIGHBOURS + 4.0) + out_bytes * rays,
            "flops": x * (17.0 * NEIGHBOURS + 12.0)}, x


def work(case):
    kind, place, M, N = case["kind"], case["place"], case["sites"], case["rays"]
    if kind == "batch":
        # expected sums of the log-uniform sizes
        mean = lambda lo, hi: (hi - lo) / math.log(hi / lo)  # noqa: E731
        m, n = mean(2_000, M), mean(10_000, N)
        w, _ = _trace_work("disk", m, n, 4.0)
        return {k: case["grids"] * v for k, v in w.items()}
    if kind == "locate":
        return {"bytes": 28.0 * N + 16.0 * M, "flops": 8.0 * 4.0 * N}
    real = 8 if case.get("precision") == "fp64" else 4
    w, x = _trace_work(place, M, N, float(real))
    if kind == "segments":
        w["bytes"] += (4.0 + real) * x + 8.0 * N
    if kind == "interact":
        w["bytes"] += 12.0 * N + 4.0 * M
    if kind == "fit":
        det, xd = _trace_work("detector", M, case["pixels"] ** 2, 4.0)
        x += xd
        w["flops"] += det["flops"] + 2.0 * x
        w["bytes"] += 52.0 * case["pixels"] ** 2 + 4.0 * M + 8.0 * (N + case["pixels"] ** 2)
    if kind == "build":
        # every cell cut by its neighbours' planes, about 30 vertices each
        w["flops"] += M * NEIGHBOURS * 30.0 * 8.0
        w["bytes"] += M * (24.0 + 56.0 + 4.0 * NEIGHBOURS)
    return w


# ---------------------------------------------------------------------------
# the same in 64 bits, every site a candidate
# ---------------------------------------------------------------------------

def _enter64(O, D, box, sphere):
    if sphere is not None:
        c, R = O.new_tensor(sphere[:3]), sphere[3]
        o = O - c
        b, q = (o * D).sum(1), (o * o).sum(1) - R * R
        disc = b * b - q
        diag = math.sqrt(sum((box[3 + i] - box[i]) ** 2 for i in range(3)))
        t = q / (torch.sqrt(disc.clamp_min(0.0)) - b) + 1e-12 * diag
        hit = (q > 0) & (b < 0) & (disc >= 0)
        return torch.where(hit[:, None], O + t[:, None] * D, O)
    lo, hi = O.new_tensor(box[:3]), O.new_tensor(box[3:])
    t1, t2 = (lo - O) / D, (hi - O) / D
    t_in = torch.minimum(t1, t2).amax(1)
    t_out = torch.maximum(t1, t2).amin(1)
    outside = ~((O >= lo) & (O <= hi)).all(1)
    hit = outside & (t_in <= t_out) & (t_out >= 0)
    P = torch.minimum(torch.maximum(O + t_in.clamp_min(0.0)[:, None] * D, lo), hi)
    return torch.where(hit[:, None], P, O)


def _nearest64(S, P):
    out = torch.empty(P.shape[0], dtype=torch.int64, device=P.device)
    step = max(1, int(5e7) // S.shape[0])
    for a in range(0, P.shape[0], step):
        d2 = P.new_zeros((P[a:a + step].shape[0], S.shape[0]))
        for c in range(3):
            d2 += (P[a:a + step, c:c + 1] - S[None, :, c]) ** 2
        out[a:a + step] = d2.argmin(1)
    return out


def _paths64(S, box, sphere, O, D):
    """(ray, cell, length, distance from the start) of every segment, in path order."""
    lo, hi = O.new_tensor(box[:3]), O.new_tensor(box[3:])
    half = 0.5 * (S * S).sum(1)
    got = []
    step = max(1, int(4e7) // S.shape[0])
    for a in range(0, O.shape[0], step):
        r, k = O[a:a + step].clone(), D[a:a + step]
        ids = torch.arange(a, a + r.shape[0], device=O.device)
        m = _nearest64(S, r)
        ok = ((r >= lo) & (r <= hi)).all(1)
        if sphere is not None:
            ok &= ((r - O.new_tensor(sphere[:3])) ** 2).sum(1) <= sphere[3] ** 2
        r, k, m, ids = r[ok], k[ok], m[ok], ids[ok]
        gone = r.new_zeros(r.shape[0])
        for _ in range(20_000):
            if ids.numel() == 0:
                break
            pm = S[m]
            den = k @ S.T - (k * pm).sum(1, keepdim=True)
            num = half[None, :] - half[m][:, None] - (r @ S.T - (r * pm).sum(1, keepdim=True))
            s = torch.where(den > 1e-15, num.clamp_min(0.0) / den, math.inf)
            s.scatter_(1, m[:, None], math.inf)
            del den, num
            best, j = s.min(1)
            if sphere is not None:
                o = r - O.new_tensor(sphere[:3])
                b, q = (k * o).sum(1), (o * o).sum(1) - sphere[3] ** 2
                w = (torch.sqrt((b * b - q).clamp_min(0.0)) - b).clamp_min(0.0)
            else:
                w = torch.where(k > 0, (hi - r) / k, torch.where(k < 0, (lo - r) / k, math.inf)).amin(1).clamp_min(0.0)
            length = torch.minimum(best, w)
            pos = length > 0
            got.append((ids[pos], m[pos], length[pos], gone[pos]))
            gone = gone + length
            r = r + length[:, None] * k
            go = best < w
            r, k, m, ids, gone = r[go], k[go], j[go], ids[go], gone[go]
    ray = torch.cat([g[0] for g in got])
    order = torch.sort(ray, stable=True)[1]
    return tuple(torch.cat([g[i] for g in got])[order] for i in range(4))


def _cheap(place, sites, rays):
    return rays * sites * (CROSSINGS[place] * sites ** (1.0 / 3.0) + 1.0) <= 4e10


def _sum_by(index, value, n):
    return torch.zeros(n, dtype=torch.float64, device=value.device).index_add_(0, index, value)


def exact(case, seed):
    kind, place = case["kind"], case["place"]
    if kind in ("batch", "locate"):
        return None
    rays = case["rays"] + (3 * case["pixels"] ** 2 if kind == "fit" else 0)
    if not _cheap(place, case["sites"], rays):
        return None
    d = _inputs(case, seed)
    O, D = d["O"], d["D"]
    N, M = O.shape[0], case["sites"]
    if case.get("enter"):
        O = _enter64(O, D, d["box"], d["sphere"])
    S = torch.from_numpy(d["sites"]).cuda()
    rho = torch.from_numpy(d["rho"]).cuda().double()
    ray, cell, length, start = _paths64(S, d["box"], d["sphere"], O, D)
    dtau = rho[cell] * length
    tau = _sum_by(ray, dtau, N)
    if kind in ("tau", "host"):
        return tau.cpu() if kind == "host" else tau
    if kind == "build":
        return [tau, None, None]
    if kind == "segments":
        return [tau, length, None, None]
    if kind == "fit":
        e = torch.exp(-tau)
        g = -2.0 * (e - d["target"].double()) * e
        return [tau, _sum_by(cell, g[ray] * length, M)]
    # interact: the running tau before each segment, capped at tau_int
    run_in = torch.cumsum(dtau, 0) - dtau
    first = torch.cat([torch.ones(1, dtype=torch.bool, device=ray.device), ray[1:] != ray[:-1]])
    base = torch.zeros(N, dtype=torch.float64, device=ray.device)
    base[ray[first]] = run_in[first]
    tin = run_in - base[ray]
    ti = d["tau_int"].double()
    a, b = torch.minimum(tin, ti[ray]), torch.minimum(tin + dtau, ti[ray])
    absorbed = _sum_by(cell, torch.exp(-a) - torch.exp(-b), M)
    s = _sum_by(ray, length, N)
    here = (tin < ti[ray]) & (tin + dtau >= ti[ray])
    s[ray[here]] = start[here] + (ti[ray[here]] - tin[here]) / rho[cell[here]]
    return [None, s, absorbed]
