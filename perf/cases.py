"""The calls whose speed is watched: binned 3- and 4-point counts of a point catalogue.

A program quantises positions, builds the neighbour graph and asks it for counts. Survey
catalogues are counted once, so for them the whole chain is one pass; a catalogue that is
queried again (other statistics, other weights) keeps its graph, and then one query is a
pass. Sizes are those of the benchmark's workloads and of the tests, or generic ones of
the same densities. Inputs are drawn on the GPU from the seed.
"""
import itertools
import math

import numpy as np
import torch

import paper_2607_06604_gb300 as gs

LATTICE = 1024  # lattice units per h^-1 Mpc
BALL = 4.0 * math.pi / 3.0


def listed():
    return [
        # the smallest calls: a light test catalogue, all of it latency and launches
        dict(name="chain_2e4", kind="chain", n=20_000, box=200.0, cat="uniform", weights="none",
             rmin=0.0, rmax=20.0, nb=10),
        # the same with weights and edges off the lattice's powers of two, in an open box
        dict(name="chain_open_odd", kind="chain", n=30_011, box=211.0, cat="clustered", open=True,
             weights="narrow", rmin=1.0, rmax=19.7, nb=9),
        # data catalogue of the benchmark's step: counts and weighted sums
        dict(name="chain_data_1e6", kind="chain", n=1_000_000, box=1000.0, cat="clustered",
             weights="narrow", rmin=0.0, rmax=40.0, nb=20),
        # its random catalogue, the largest call of the step
        dict(name="chain_randoms_3e6", kind="chain", n=3_000_000, box=1000.0, cat="uniform",
             weights="narrow", rmin=0.0, rmax=40.0, nb=20),
        # BAO scales: wide bins, rows of thousands of neighbours, edges kept in host memory
        # under a device budget and streamed in windows
        dict(name="bao_windows", kind="windows", n=60_000, box=585.0, cat="clustered", open=True,
             sigma=5.0, weights="none", rmin=0.0, rmax=150.0, nb=15, windows=3),
        # a mock ensemble that is resident: many uneven catalogues counted in one launch
        dict(name="mocks_batch", kind="batch", n=50_000, n2=120_000, count=3, box=500.0,
             cat="lognormal", weights="none", rmin=0.0, rmax=60.0, nb=12),
        # parity-decomposed 4pCF with the 2pCF and the disconnected term on the same graph
        dict(name="parity_2e5", kind="parity", n=200_000, box=400.0, cat="clustered",
             weights="none", rmin=0.0, rmax=30.0, nb=8),
        # 4pCF of one mock of an ensemble, built and counted (plain channel, few bins)
        dict(name="mock_4pcf", kind="chain4", n=100_003, box=500.0, cat="lognormal",
             weights="none", rmin=0.0, rmax=25.0, nb=6),
        # parity channel from pixelised spoke directions
        dict(name="pixel_1e5", kind="pixel", n=100_000, box=317.0, cat="clustered",
             weights="none", rmin=0.0, rmax=30.0, nb=8),
        # connected 4pCF: data and randoms 1:1, signed weights, two weighted 4pCF passes
        dict(name="connected_1e5", kind="connected", n=50_000, box=317.0, cat="clustered",
             weights="narrow", rmin=0.0, rmax=30.0, nb=8),
        # anisotropic 3pCF of randoms
        dict(name="mu_1e6", kind="mu", n=1_000_000, box=693.0, cat="uniform", weights="none",
             rmin=0.0, rmax=40.0, nb=20, nmu=10),
        # equilateral 3pCF and weighted 2pCF of a kept graph
        dict(name="equi_pairs_1e6", kind="equi", n=1_000_000, box=693.0, cat="uniform",
             weights="narrow", rmin=0.0, rmax=40.0, nb=20),
    ]


# kind -> (smallest n, largest n, smallest and largest mean number of neighbours, most
# n * neighbours^p of a pass, p, smallest and largest nb)
_RANGES = {
    "chain": (5_000, 2_500_000, 30, 1500, 1.2e12, 2, 4, 24),
    "windows": (20_000, 80_000, 400, 3500, 6e11, 2, 8, 18),
    "batch": (10_000, 150_000, 60, 1500, 3e11, 2, 6, 16),
    "parity": (5_000, 200_000, 30, 350, 6e12, 3, 3, 9),
    "chain4": (5_000, 150_000, 30, 300, 3e12, 3, 3, 9),
    "pixel": (5_000, 100_000, 30, 350, 3e12, 3, 3, 8),
    "connected": (4_000, 50_000, 30, 300, 1e12, 3, 3, 8),
    "mu": (10_000, 1_500_000, 50, 900, 5e11, 2, 5, 20),
    "equi": (10_000, 1_500_000, 50, 900, 5e11, 2, 5, 24),
}


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["chain", "chain", "chain"] + [k for k in _RANGES if k != "chain"])
    n0, n1, k0, k1, most, p, nb0, nb1 = _RANGES[kind]
    n = int(_log(rng, n0, n1))
    # a periodic box is more than four times rmax wide: n > 64 / BALL neighbours
    k = _log(rng, k0, max(k0, min(k1, n / 18.0, (most / n) ** (1.0 / p))))
    rho = _log(rng, 3e-4, 4e-3)
    rmax = round((k / (BALL * rho)) ** (1.0 / 3.0), 2)
    rmax = min(rmax, 300.0)
    c = dict(kind=kind, n=n, box=float(max(math.ceil((n / rho) ** (1.0 / 3.0)),
                                           math.ceil(4.1 * rmax))),
             nb=rng.randint(nb0, nb1), rmax=rmax,
             rmin=rng.choice([0.0, 0.0, 0.0, round(0.1 * rmax, 1)]))
    c["cat"] = rng.choice(["uniform", "clustered"])
    c["weights"] = "none"
    if kind == "chain":
        c["weights"] = rng.choice(["none", "narrow", "narrow"] + ["wide"] * (n * k * k < 2e11))
        c["open"] = rng.random() < 0.3
    elif kind in ("connected", "equi"):
        c["weights"] = "narrow"
    elif kind == "windows":
        c.update(open=True, cat="clustered", sigma=5.0, windows=rng.randint(2, 5))
    elif kind == "batch":
        c.update(cat="lognormal", n2=int(_log(rng, n0, n)), count=rng.randint(2, 4))
    elif kind == "chain4":
        c["cat"] = "lognormal"
    elif kind == "mu":
        c["nmu"] = rng.randint(4, 16)
    return c


def _edges(c):
    return np.array([math.floor(LATTICE * (c["rmin"] + b * (c["rmax"] - c["rmin"]) / c["nb"]) + 0.5)
                     for b in range(c["nb"] + 1)], dtype=np.int64)


def _rand(*shape, g):
    return torch.rand(*shape, generator=g, device="cuda", dtype=torch.float64)


def _catalogue(cat, n, box, g, sigma=2.0, wrap=True):
    """Positions in [0, box)^3: uniform, a Neyman-Scott process of ten points per parent,
    or a lognormal field on a 128^3 grid."""
    if cat == "uniform":
        return _rand(n, 3, g=g) * box
    if cat == "clustered":
        parents = _rand(max(1, n // 10), 3, g=g) * box
        at = torch.randint(parents.shape[0], (n,), generator=g, device="cuda")
        off = torch.randn(n, 3, generator=g, device="cuda", dtype=torch.float64) * sigma
        x = parents[at] + off
        if wrap:
            x = torch.remainder(x, box)
        else:  # reflected at the faces of an open box
            x = x.abs()
            x = torch.where(x >= box, 2 * box - x, x)
        return x.clamp_(0.0, box * (1 - 1e-9))
    m = 128
    white = torch.randn(m, m, m, generator=g, device="cuda")
    f = 2 * math.pi * torch.fft.fftfreq(m, d=box / m, device="cuda")
    fz = 2 * math.pi * torch.fft.rfftfreq(m, d=box / m, device="cuda")
    k2 = f[:, None, None] ** 2 + f[None, :, None] ** 2 + fz[None, None, :] ** 2
    amp = torch.where(k2 > 0, k2 ** -0.375, torch.zeros_like(k2)) * torch.exp(-2.0 * k2)
    field = torch.fft.irfftn(torch.fft.rfftn(white) * amp, s=(m, m, m))
    dens = torch.exp((field - field.mean()) / field.std()).double().flatten()
    cum = torch.cumsum(dens, 0)
    cell = torch.searchsorted(cum, _rand(n, g=g) * cum[-1]).clamp_(max=m ** 3 - 1)
    xyz = torch.stack([cell // (m * m), (cell // m) % m, cell % m], 1).double()
    return ((xyz + _rand(n, 3, g=g)) * (box / m)).clamp_(0.0, box * (1 - 1e-9))


def _weights(kind, n, g):
    """FP32 weights: U(0.5, 1.5), or spread over a factor of a thousand."""
    u = _rand(n, g=g)
    if kind == "none":
        return None
    return ((0.5 + u) if kind == "narrow" else torch.exp2(10.0 * u - 9.0)).float()


def _quantised(c, pos):
    return gs.gs_quantize(pos, c["box_u"], not c.get("open", False))


def _build(c, xyz, **opts):
    return gs.gs_build_graph(xyz, 0 if c.get("open") else c["box_u"], c["edges"], **opts)


def prepare(case, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    c = dict(case, box_u=int(round(case["box"] * LATTICE)), edges=_edges(case))
    st = {"c": c}
    ns = [case["n"]]
    if case["kind"] == "batch":
        lo, hi = sorted((case["n"], case["n2"]))
        ns = [int(lo + (hi - lo) * k / (case["count"] - 1)) for k in range(case["count"])]
    pos = [_catalogue(case["cat"], n, case["box"], g, case.get("sigma", 2.0),
                      not case.get("open", False)) for n in ns]
    st["w"] = _weights(case["weights"], ns[0], g)
    st["like"] = torch.empty(0, device="cuda")
    if case["kind"] in ("chain", "chain4"):
        st["pos"] = pos[0]
    elif case["kind"] == "connected":
        rand = _catalogue("uniform", case["n"], case["box"], g)
        wr = _weights("narrow", case["n"], g)
        wd, wr = st["w"].double() / st["w"].double().sum(), wr.double() / wr.double().sum()
        st["w"] = torch.cat([wd, -wr]).float()
        st["wr"] = wr.float()
        st["xyz"] = _quantised(c, torch.cat([pos[0], rand]))
        st["graph"] = _build(c, st["xyz"])
        st["graph_r"] = _build(c, _quantised(c, rand))
    elif case["kind"] == "batch":
        st["graphs"] = [_build(c, _quantised(c, p)) for p in pos]
    else:
        st["xyz"] = _quantised(c, pos[0])
        st["graph"] = _build(c, st["xyz"], force_windows=case.get("windows", 0))
    torch.cuda.synchronize()
    return st


def run(st):
    c, w, like = st["c"], st["w"], st["like"]
    kind = c["kind"]
    if kind == "chain":
        graph = _build(c, _quantised(c, st["pos"]))
        out = gs.gs_count_3pcf(graph, w, like=like)
        gs.gs_free_graph(graph)
        return {"counts": out} if w is None else {"counts": out[0], "wsum": out[1]}
    if kind == "chain4":
        graph = _build(c, _quantised(c, st["pos"]))
        out = gs.gs_count_4pcf(graph, like=like)
        gs.gs_free_graph(graph)
        return {"counts": out}
    if kind == "windows":
        return {"counts": gs.gs_count_3pcf(st["graph"], like=like)}
    if kind == "batch":
        return {"counts": [o[0] for o in gs.gs_count_3pcf_batch(st["graphs"], like=like)]}
    if kind == "parity":
        even, odd = gs.gs_count_4pcf_parity(st["graph"], like=like)
        pairs, xi, zeta = gs.gs_disconnected_4pcf(st["graph"], like=like)
        return {"even": even, "odd": odd, "pairs": pairs, "xi": xi, "zeta_disc": zeta}
    if kind == "pixel":
        even, odd = gs.gs_count_4pcf_parity_pix(st["graph"], like=like)
        return {"even": even, "odd": odd}
    if kind == "connected":
        return gs.gs_connected_4pcf(st["graph"], w, st["graph_r"], st["wr"])
    if kind == "mu":
        return {"counts": gs.gs_count_3pcf_mu(st["graph"], c["nmu"], like=like)}
    if kind == "equi":
        counts, wsum = gs.gs_count_3pcf_equilateral(st["graph"], w)
        pairs, xi, _ = gs.gs_disconnected_4pcf(st["graph"], w, zeta=False)
        return {"counts": counts, "wsum": wsum, "pairs": pairs, "xi": xi}
    raise ValueError(kind)


def _orbits(nb):
    return (nb ** 6 + 9 * nb ** 4 + 14 * nb ** 2) // 24


def work(case):
    """Bytes: positions or the stored edges (4 B) and weights in, counts out. Operations: a
    distance (8) for each of the tuple's pairs that the hub's edges do not give already, for
    the tuples of a uniform catalogue of this density (15/32 of a ball's point pairs, and a
    fifth of its triples, lie within the radius of one another)."""
    n, nb, kind = case["n"], case["nb"], case["kind"]
    if kind == "batch":
        m = case["count"]
        n, ns = None, [case["n"] + (case["n2"] - case["n"]) * k / (m - 1) for k in range(m)]
    elif kind == "connected":
        ns = [2 * n, n]
    else:
        ns = [n]
    ball = BALL * case["rmax"] ** 3 / case["box"] ** 3
    edges = sum(x * x * ball / 2 for x in ns)
    tri = sum(x * (x * ball) ** 2 / 6 * 15 / 32 for x in ns)
    tet = sum(x * (x * ball) ** 3 / 24 / 5 for x in ns)
    nc3 = nb * (nb + 1) * (nb + 2) // 6
    points = sum(ns)
    if kind == "chain":
        wide = 12 if case["weights"] != "none" else 0
        return {"bytes": 24 * points + wide / 3 * points + (8 + (wide and 8)) * nc3,
                "flops": 8 * tri + 8 * edges}
    if kind == "chain4":
        return {"bytes": 24 * points + 8 * _orbits(nb), "flops": 24 * tet + 8 * tri}
    if kind in ("windows", "batch"):
        return {"bytes": 4 * edges + 16 * points + 8 * nc3 * len(ns), "flops": 8 * tri}
    if kind in ("parity", "pixel"):
        return {"bytes": 4 * edges + 16 * points + 24 * _orbits(nb), "flops": 24 * tet + 8 * tri}
    if kind == "connected":
        return {"bytes": 4 * edges + 20 * points + 32 * _orbits(nb), "flops": 27 * tet + 8 * tri}
    if kind == "mu":
        return {"bytes": 4 * edges + 16 * points + 8 * nc3 * (case["nmu"] + 1), "flops": 24 * tri}
    # one bin's share of the triangles for the equilateral ones; every edge for the pairs
    return {"bytes": 4 * edges + 20 * points + 32 * nb, "flops": 8 * tri / nb + 3 * edges}


# ---- plain 64-bit values -------------------------------------------------------------


def _pair_bins(x, box_u, e2, lo, hi):
    """Squared distances of points lo..hi to all points as bins (-1: no edge)."""
    d2 = torch.zeros(hi - lo, x.shape[0], dtype=torch.int64, device=x.device)
    for a in range(3):
        d = (x[None, :, a] - x[lo:hi, a, None]).abs()
        if box_u:
            d = torch.minimum(d, box_u - d)
        d2 += d * d
    b = torch.bucketize(d2, e2, right=True) - 1
    return torch.where(b < e2.numel() - 1, b, torch.full_like(b, -1))


def _pair_sums(x, box_u, e2, w):
    """Sum of w_i w_j (and the number) of the unordered pairs in each bin."""
    nb, n = e2.numel() - 1, x.shape[0]
    num = torch.zeros(nb + 1, dtype=torch.float64, device=x.device)
    cnt = torch.zeros(nb + 1, dtype=torch.float64, device=x.device)
    step = max(1, 100_000_000 // n)
    for lo in range(0, n, step):
        hi = min(n, lo + step)
        b = _pair_bins(x, box_u, e2, lo, hi)
        b[torch.arange(hi - lo, device=x.device), torch.arange(lo, hi, device=x.device)] = -1
        for k in range(nb):
            m = b == k
            cnt[k] += m.sum()
            if w is not None:
                num[k] += (w[lo:hi] * (m.double() @ w)).sum()
    return (num if w is not None else cnt)[:nb] / 2


def _rr(c, w):
    """Analytic random pairs of a periodic box."""
    p = c["n"] * (c["n"] - 1) / 2 if w is None else float((w.sum() ** 2 - (w * w).sum()) / 2)
    e = c["edges"].astype(np.float64)
    return p * (4.0 * math.pi / 3.0) * (e[1:] ** 3 - e[:-1] ** 3) / float(c["box_u"]) ** 3


def _reps(nb):
    """Smallest member of every class of edge-bin tuples (01, 02, 03, 12, 13, 23) under
    relabelling of the four vertices, in ascending order."""
    slots = list(itertools.combinations(range(4), 2))
    t = np.indices((nb,) * 6).reshape(6, -1)
    power = nb ** np.arange(5, -1, -1)
    best = None
    for p in itertools.permutations(range(4)):
        src = [slots.index(tuple(sorted((p[a], p[b])))) for a, b in slots]
        code = power @ t[src]
        best = code if best is None else np.minimum(best, code)
    own = power @ t
    return t[:, own == best]


def _disconnected(xi, nb):
    r = _reps(nb)
    return xi[r[0]] * xi[r[5]] + xi[r[1]] * xi[r[4]] + xi[r[2]] * xi[r[3]]


def _triangles(x, box_u, e2, w):
    """Weighted triangle sums per sorted bin triple, hub by hub in blocks."""
    nb, n = e2.numel() - 1, x.shape[0]
    bins = torch.empty(n, n, dtype=torch.int8, device=x.device)
    for lo in range(0, n, 2000):
        bins[lo:lo + 2000] = _pair_bins(x, box_u, e2, lo, min(n, lo + 2000)).to(torch.int8)
    bins.fill_diagonal_(-1)
    rank = {t: k for k, t in enumerate(itertools.combinations_with_replacement(range(nb), 3))}
    table = torch.tensor([rank[tuple(sorted(t))] for t in itertools.product(range(nb), repeat=3)],
                         device=x.device)
    out = torch.zeros(len(rank), dtype=torch.float64, device=x.device)
    w = w.double()
    for i in range(n - 2):
        near = torch.nonzero(bins[i, i + 1:] >= 0).squeeze(1) + i + 1
        own, wn = bins[i, near].long(), w[near]
        bjk = bins[near][:, near].long()
        at = (own[:, None] * nb + own[None, :]) * nb + bjk
        ok = torch.triu(bjk >= 0, 1)
        out += w[i] * torch.bincount(table[at.clamp_(min=0)].flatten(), minlength=len(rank),
                                     weights=(wn[:, None] * wn[None, :] * ok).flatten())
    return out.cpu().numpy()


def exact(case, seed):
    kind, n = case["kind"], case["n"]
    near = n * BALL * case["rmax"] ** 3 / case["box"] ** 3
    if not (kind in ("parity", "connected")) and not (kind == "equi" and n <= 120_000) and \
       not (kind == "chain" and case["weights"] != "none" and n <= 31_000 and n * near ** 2 < 3e9):
        return None
    st = prepare(case, seed)
    c = st["c"]
    box_u = 0 if case.get("open") else c["box_u"]
    e2 = torch.from_numpy(c["edges"] ** 2).cuda()
    if kind == "chain":
        x = torch.floor(st["pos"] * LATTICE).long()
        if box_u:
            x = torch.remainder(x, box_u)
        return {"counts": None, "wsum": _triangles(x, box_u, e2, st["w"])}
    x = st["xyz"].long()
    w = None if st["w"] is None else st["w"].double()
    sums = _pair_sums(x, box_u, e2, w).cpu().numpy()
    if kind == "parity":
        xi = sums / _rr(c, None) - 1
        return {"even": None, "odd": None, "pairs": None, "xi": xi,
                "zeta_disc": _disconnected(xi, case["nb"])}
    if kind == "equi":
        return {"counts": None, "wsum": None, "pairs": None, "xi": sums / _rr(c, w) - 1}
    xi = sums / _pair_sums(x[n:], box_u, e2, st["wr"].double()).cpu().numpy()
    return {"xi": xi, "zeta_even": None, "zeta_odd": None,
            "zeta_disc": _disconnected(xi, case["nb"]), "zeta_conn": None}
