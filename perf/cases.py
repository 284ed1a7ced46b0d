"""Timed cases of the spatial-statistics library: what a user's program has it do.

A program holds one cell grid (or batch) per cloud size, and for every cloud, reconstruction or
relabelling it builds the grid and runs a statistic.  One pass is that: build and query, on device
tensors, through the Python binding.  The clouds are the synthetic specimens of the paper's
benchmarks (Poisson cylinders of 40 ions/nm^3, precipitate needles of 30 ions/nm^3), the
parameters those of the benchmark and of the tests.

Kinds of case
  stat     exact RDF + kNN histograms (build + spatstat per type combination), optionally with
           per-ion outputs, the g(r) normalisation, or labels randomised before the build
  soft     one step of a fit through the smoothed RDF: forward, loss, gradients of the positions
           and of the scale ("autograd": torch.autograd through soft_rdf; "handle": the forward and
           adjoint calls on a grid that the program keeps)
  sdm      spatial distribution map
  cluster  maximum-separation clustering
  batch    many regions of interest, a whole parameter sweep each
"""
import math

import numpy as np
import torch

import paper_2004_05188_gb300 as ps
from paper_2004_05188_gb300 import specimen

COMBOS = {"all-all": ("all", "all"), "Sc-Sc": ([1], [1]), "Si-Si": ([2], [2]), "Al-Sc": ([0], [1]),
          "all-Sc": ("all", [1])}
# expected type fractions; the needle's Sc: 0.3 % of the matrix and 25 % of the precipitates
# (1e-3 /nm^3, log-normal radii: mean volume 4/3 pi 2^3 exp(4.5 * 0.3^2) nm^3)
PREC_SHARE = 1e-3 * 4.0 / 3.0 * math.pi * 8.0 * math.exp(4.5 * 0.09)
FRACTION = {"cylinder": {0: 0.97, 1: 0.02, 2: 0.01},
            "needle": {0: 0.95, 1: 0.003 + 0.25 * PREC_SHARE, 2: 0.002}}
DENSITY = {"cylinder": 40.0, "needle": 30.0}
SOFT_SIGMA = 0.05
BATCH_BINS, BATCH_RMAX, BATCH_DSRF, BATCH_K = (0.0, 0.01, 300), [100, 200, 300], [0.0, 1.0, 2.0], 20
BATCH_PAIRS = [("all", "all"), ([1], [1]), ([0], [1])]


def _stat(name, cloud, n, combos, ks, stop, dsrf, cell=1.0, split="0", rdf=True, per_central=False, gr=False,
          shuffle=False):
    c = {"kind": "stat", "cloud": cloud, "n": n, "combos": combos, "ks": ks, "stop": stop, "step": 0.01, "dsrf": dsrf,
         "cell": cell, "split": split, "rdf": rdf, "per_central": per_central, "gr": gr, "shuffle": shuffle}
    return dict(c, name=name) if name else c


def _soft(name, cloud, n, form, cell):
    c = {"kind": "soft", "cloud": cloud, "n": n, "form": form, "cell": cell, "step": 0.02, "stop": 2.0, "dsrf": 2.3}
    return dict(c, name=name) if name else c


def _sdm(name, cloud, n, combo, n_vox, w, cell):
    c = {"kind": "sdm", "cloud": cloud, "n": n, "combos": combo, "stop": 2.0, "n_vox": n_vox, "w": w, "dsrf": 2.0,
         "cell": cell}
    return dict(c, name=name) if name else c


def _cluster(name, cloud, n, types, d_max):
    c = {"kind": "cluster", "cloud": cloud, "n": n, "combos": types, "stop": d_max, "n_min": 5, "dsrf": 2.0}
    return dict(c, name=name) if name else c


def _batch(name, rois, lo, hi, cell):
    c = {"kind": "batch", "rois": rois, "lo": lo, "hi": hi, "cell": cell}
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest call: one region of interest of a few ten thousand ions, as the library's
        # smoke check runs it, with the normalised g(r); launches and latency count
        _stat("roi_20k", "cylinder", 20_000, "all-all", "1,4", 1.5, 1.0, gr=True),
        # the paper's small specimen, on the configuration that the autotuner picks for it
        _stat("cylinder_200k", "cylinder", 200_000, "all-all", "1", 2.0, 1.0, cell=1 / 3, split="1"),
        # default options and the per-ion results (k-th distances, in-range counts) of an odd-sized
        # cloud: what an analysis that maps the neighbourhoods back onto the ions asks for
        _stat("cylinder_100k_per_ion", "cylinder", 100_003, "all-all", "1,4,10", 2.0, 0.5, per_central=True),
        # solute statistics of a needle: sparse types, default options; the grid builds count
        _stat("needle_8m_solutes", "needle", 8_066_977, "Sc-Sc+Si-Si", "1,5,10", 2.0, 2.0),
        # matrix ions about solutes with randomised labels, the reference that the paper computes
        # beside every statistic: many centrals that are not among the neighbours
        _stat("needle_3m_al_sc_random", "needle", 3_000_017, "Al-Sc", "1,5,10", 2.0, 2.0, shuffle=True),
        # all ions of the needle: dense, bound by the pair tests
        _stat("needle_8m_all", "needle", 8_066_977, "all-all", "10", 2.0, 2.0, cell=0.5, split="1"),
        # the full-scale needle's statistics (all-all in passes, Sc-Sc in one pass, one grid), 1/20 of
        # its ions
        _stat("needle_100m", "needle", 100_000_000, "all-all+Sc-Sc", "10", 2.0, 2.0, cell=0.5, split="1,0"),
        # a step of a fit through the smoothed RDF, through autograd, on the small specimen
        _soft("soft_200k_autograd", "cylinder", 200_000, "autograd", 1.0),
        # the same on the 1e7-ion needle, with a grid that the program keeps
        _soft("soft_10m", "needle", 10_000_000, "handle", 0.5),
        # spatial distribution map with the paper's setting (2 nm, voxels of 0.025 nm), all ions
        _sdm("sdm_8m_all", "needle", 8_066_977, "all-all", 160, 0.025, 1.0),
        # solute clusters of the needle, one run of the paper's d_max sweep
        _cluster("cluster_8m_sc", "needle", 8_066_977, "Sc-Sc", 0.5),
        # a sensitivity study: regions of uneven size, k = 1..20, three r_max, three d_srf thresholds
        # and three type pairs each, in one call
        _batch("batch_24_rois", 24, 10_000, 300_000, 0.5),
    ]


def _log(rng, lo, hi):
    return int(round(lo * (hi / lo) ** rng.random()))


def draw(rng):
    u = rng.random()
    cloud = rng.choice(["cylinder", "needle"])
    if u < 0.5:
        cell, split = rng.choice([(1.0, "0"), (1.0, "0"), (0.5, "1"), (1 / 3, "1"), (0.5, "0"), (0.75, "0")])
        combos = rng.choice(["all-all", "all-all", "Sc-Sc", "Al-Sc", "all-Sc", "Sc-Sc+Si-Si"])
        k = rng.choice(["1", "10", "1,5,10", "2,20", "32", ""])
        n = _log(rng, 12_000, 3_000_000 if "all-all" in combos else 20_000_000)
        per = rng.random() < 0.2 and n < 2_000_000
        return _stat(None, cloud, n, combos, k, rng.choice([1.0, 1.5, 2.0]), rng.choice([0.0, 1.0, 2.0]), cell, split,
                     rdf=k == "" or rng.random() < 0.85, per_central=per, gr=rng.random() < 0.3,
                     shuffle=rng.random() < 0.25)
    if u < 0.7:
        n = _log(rng, 30_000, 3_000_000)
        return _soft(None, cloud, n, rng.choice(["autograd", "handle"]), rng.choice([1.0, 0.5]))
    if u < 0.8:
        combo = rng.choice(["all-all", "Sc-Sc", "Al-Sc"])
        n_vox, w = rng.choice([(160, 0.025), (80, 0.05), (81, 0.05), (33, 0.12)])
        n = _log(rng, 30_000, 2_000_000 if combo == "all-all" else 8_000_000)
        return _sdm(None, cloud, n, combo, n_vox, w, rng.choice([1.0, 0.5]))
    if u < 0.9:
        types = rng.choice(["Sc-Sc", "Si-Si", "all-all"])
        n = _log(rng, 30_000, 10_000_000)
        d_max = round(rng.uniform(0.1, 0.15) if types == "all-all" else rng.uniform(0.1, 0.7), 3)
        return _cluster(None, cloud, n, types, d_max)
    return _batch(None, rng.randint(3, 24), 10_000, _log(rng, 20_000, 300_000), rng.choice([1.0, 0.5]))


# ---------------------------------------------------------------------------------------------
# clouds
# ---------------------------------------------------------------------------------------------

def _shape(cloud, n):
    """(radius, half-angle, height) of a specimen of n expected ions.  Up to 2e7 ions the needle is
    the 8e6-ion one scaled, above that the full-scale needle (tip 40 nm, 15 deg) cut at n ions."""
    if cloud == "cylinder":
        R = (n / (DENSITY["cylinder"] * math.pi * 1.59)) ** (1.0 / 3.0)
        return R, 0.0, 1.59 * R
    if n <= 20_000_000:
        f = (n / (DENSITY["needle"] * specimen.frustum_volume(20.0, 10.0, 100.0))) ** (1.0 / 3.0)
        return 20.0 * f, 10.0, 100.0 * f
    return 40.0, 15.0, specimen.height_for(n, 40.0, 15.0)


def _cloud(case, seed):
    """The cloud of exactly n ions; a needle (whose ion count depends on the seed) is made a little
    longer and cut at its base."""
    n = case["n"]
    if case["cloud"] == "cylinder":
        r, _, h = _shape("cylinder", n)
        a = specimen.cylinder(seed, n, r, h, (0.97, 0.02, 0.01))
    else:
        layers = _shape("needle", n)[2] / specimen.FCC_A
        grow = n * (1.0 + 2.0 / layers) + 6.0 * math.sqrt(n)
        a = (np.empty(0),)
        while a[0].shape[0] < n:
            r, ang, h = _shape("needle", grow)
            a = specimen.needle(specimen.needle_params(r, ang, h, seed))
            grow *= 1.02
    return tuple(torch.from_numpy(x[:n]).cuda() for x in a)


def _volume(cloud, n):
    r, ang, h = _shape(cloud, n)
    return specimen.frustum_volume(r, ang, h)


def _bins(case):
    return ps.bins_from_spec(0.0, case["step"], case["stop"])


def _ks(case):
    return [int(k) for k in case["ks"].split(",") if k]


# ---------------------------------------------------------------------------------------------
# what a program has in hand, and one pass
# ---------------------------------------------------------------------------------------------

def prepare(case, seed):
    if case["kind"] == "batch":
        rng = np.random.default_rng(seed)
        rois = []
        for i in range(case["rois"]):
            n = int(round(case["lo"] * (case["hi"] / case["lo"]) ** rng.random()))
            rois.append(tuple(torch.from_numpy(a).cuda() for a in specimen.roi(i, n, seed0=1000 * (seed % 100_003))))
        return {"case": case, "batch": ps.Batch(rois, BATCH_BINS, BATCH_RMAX, BATCH_DSRF, BATCH_PAIRS, BATCH_K,
                                                case["cell"])}
    X, T, D = _cloud(case, seed)
    s = {"case": case, "X": X, "T": T, "D": D, "seed": seed}
    n = X.shape[0]
    if case["kind"] == "stat":
        s["grid"] = ps.Grid(n, case["cell"], 0, case["split"][0] == "1")
        s["volume"] = _volume(case["cloud"], case["n"])
    elif case["kind"] == "soft":
        bins = _bins(case)
        # factor: smoothed counts -> g(r) at the cloud's mean density; target: an oscillating g(r)
        e = torch.arange(bins[2] + 1, dtype=torch.float64) * bins[1]
        shell = 4.0 / 3.0 * math.pi * (e[1:] ** 3 - e[:-1] ** 3)
        n_c = int((D >= case["dsrf"]).sum())
        rho = n / _volume(case["cloud"], case["n"])
        mid = 0.5 * (e[1:] + e[:-1])
        s["factor"] = (1.0 / (max(n_c, 1) * rho * shell)).float().cuda()
        s["target"] = (1.0 + 0.5 * torch.cos(2.0 * math.pi * mid / 0.286)).float().cuda()
        if case["form"] == "handle":
            s["grid"] = ps.Grid(n, case["cell"])
        else:
            X.requires_grad_(True)
            s["scale"] = torch.ones(1, requires_grad=True)
    else:
        s["grid"] = ps.Grid(n, case.get("cell", 1.0))
    return s


def run(s):
    return {"stat": _run_stat, "soft": _run_soft, "sdm": _run_sdm, "cluster": _run_cluster,
            "batch": lambda s: s["batch"].run()}[s["case"]["kind"]](s)


def _run_stat(s):
    case, g = s["case"], s["grid"]
    bins, ks, combos = _bins(case), _ks(case), case["combos"].split("+")
    splits = case["split"].split(",")
    r_cut = case["stop"] * (1.0 + 1e-6)
    T = ps.shuffle_labels(s["T"], s["seed"]) if case["shuffle"] else s["T"]
    outs = []
    for i, name in enumerate(combos):
        ctr, nbr = COMBOS[name]
        if len(splits) > 1:
            g.set_query_opts(split=splits[i] == "1")
        g.build(s["X"], T, nbr, r_cut)
        out = ps.spatstat(g, s["D"], ctr, case["dsrf"], bins, ks, rdf=case["rdf"], per_central=case["per_central"],
                          check=False)
        if case["gr"] and case["rdf"]:
            out["g"] = ps.rdf_normalise(g, out["meta"], bins, s["volume"], rdf=out["rdf"])[0]
        outs.append(out)
    return outs


def _run_soft(s):
    case, X, T, D = s["case"], s["X"], s["T"], s["D"]
    bins = _bins(case)
    if case["form"] == "autograd":
        X.grad = s["scale"].grad = None
        h = ps.soft_rdf(X, s["scale"], T, D, "all", "all", case["dsrf"], SOFT_SIGMA, bins)
        loss = ((h * s["factor"] - s["target"]) ** 2).sum()
        loss.backward()
        return {"h": h.detach(), "grad": X.grad, "grad_scale": s["scale"].grad}
    g = s["grid"].build(X, T, "all", ps.soft_r_cut(bins, SOFT_SIGMA, 1.0))
    h = ps.soft_rdf_fwd(g, D, "all", case["dsrf"], SOFT_SIGMA, 1.0, bins)
    G = 2.0 * (h * s["factor"] - s["target"]) * s["factor"]
    grad, grad_scale = ps.soft_rdf_bwd(g, D, "all", case["dsrf"], SOFT_SIGMA, 1.0, bins, G)
    return {"h": h, "grad": grad, "grad_scale": grad_scale}


def _run_sdm(s):
    case = s["case"]
    ctr, nbr = COMBOS[case["combos"]]
    g = s["grid"].build(s["X"], s["T"], nbr, case["stop"])
    return ps.sdm(g, s["D"], ctr, case["dsrf"], case["stop"], case["w"], case["n_vox"])


def _run_cluster(s):
    case = s["case"]
    g = s["grid"].build(s["X"], s["T"], COMBOS[case["combos"]][1], case["stop"] * (1.0 + 1e-6))
    return ps.cluster(g, s["D"], case["stop"], case["n_min"], case["dsrf"], 1024)


# ---------------------------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------------------------

PAIR_FLOPS = 9       # 3 sub, 3 mul, 2 add, 1 compare
SOFT_PAIR_FLOPS = 60  # forward: distance and moments; adjoint: distance, weight, three components, both ends


def _central_share(cloud, n, dsrf):
    r, ang, h = _shape(cloud, n)
    if cloud == "cylinder":
        return max(0.0, r - dsrf) ** 2 * max(0.0, h - 2 * dsrf) / (r * r * h)
    t = math.tan(math.radians(ang))
    hi, top = h - 2 * dsrf, r + dsrf * t - dsrf / math.cos(math.radians(ang))
    if hi <= 0 or top <= 0:
        return 0.0
    return specimen.frustum_volume(top, ang, hi) / specimen.frustum_volume(r, ang, h)


def _share(cloud, types):
    return 1.0 if types == "all" else sum(FRACTION[cloud][t] for t in types)


def _pairs(cloud, n, combo, radius, dsrf):
    """In-range pairs that have to be tested: each unordered pair once where the centrals are neighbours."""
    ctr, nbr = COMBOS[combo]
    near = DENSITY[cloud] * 4.0 / 3.0 * math.pi * radius ** 3
    per = near * _share(cloud, nbr)
    if cloud == "needle" and combo == "Sc-Sc":  # most Sc sits in precipitates
        per = near * 0.25 * 0.4
    same = nbr == "all" or (ctr != "all" and set(ctr) <= set(nbr))
    return n * _share(cloud, ctr) * _central_share(cloud, n, dsrf) * per * (0.5 if same else 1.0)


def work(case):
    if case["kind"] == "batch":
        rec = BATCH_BINS[2] * (1 + BATCH_K) + 4 + 2 * BATCH_K
        out = case["rois"] * len(BATCH_PAIRS) * len(BATCH_RMAX) * len(BATCH_DSRF) * rec * 8
        mean = (case["hi"] - case["lo"]) / math.log(case["hi"] / case["lo"])
        n = int(case["rois"] * mean)
        pairs = 0.5 * sum(_pairs(c, mean, "all-all", 3.0, 0.0) * case["rois"] for c in ("needle", "cylinder"))
        return {"bytes": 17 * n + out, "flops": PAIR_FLOPS * pairs}
    n, cloud = case["n"], case["cloud"]
    if case["kind"] == "soft":
        pairs = _pairs(cloud, n, "all-all", case["stop"] + 6 * SOFT_SIGMA, case["dsrf"])
        return {"bytes": 17 * n + 12 * n, "flops": SOFT_PAIR_FLOPS * pairs}
    if case["kind"] == "sdm":
        return {"bytes": 17 * n + 8 * case["n_vox"] ** 3,
                "flops": PAIR_FLOPS * _pairs(cloud, n, case["combos"], case["stop"], case["dsrf"])}
    if case["kind"] == "cluster":
        return {"bytes": 17 * n + 4 * n, "flops": PAIR_FLOPS * _pairs(cloud, n, case["combos"], case["stop"], 0.0)}
    ks, combos = _ks(case), case["combos"].split("+")
    nb = _bins(case)[2]
    flops = sum(PAIR_FLOPS * _pairs(cloud, n, c, case["stop"], case["dsrf"]) for c in combos)
    per = (4 * len(ks) + 4) * n if case["per_central"] else 0
    return {"bytes": 17 * n + len(combos) * (8 * nb * (1 + len(ks)) + per), "flops": flops}


# ---------------------------------------------------------------------------------------------
# the computed numbers in 64 bits
# ---------------------------------------------------------------------------------------------

EXACT_STAT_MAX, EXACT_SOFT_MAX = 130_000, 250_000


def _in_set(T, types):
    if types == "all":
        return torch.ones_like(T, dtype=torch.bool)
    return sum((T == t) for t in types).bool()


def _d2_rows(P, Q):
    """Squared distances [len(P), len(Q)], float64."""
    d2 = torch.zeros((P.shape[0], Q.shape[0]), dtype=torch.float64, device=P.device)
    for ax in range(3):
        d2 += (P[:, ax, None] - Q[None, :, ax]) ** 2
    return d2


def exact(case, seed):
    if case["kind"] == "stat" and not case["shuffle"] and case["n"] <= EXACT_STAT_MAX:
        return _exact_stat(case, seed)
    if case["kind"] == "soft" and case["n"] <= EXACT_SOFT_MAX:
        return _exact_soft(case, seed)
    return None


def _exact_stat(case, seed):
    """kth distances (squared) and g(r) of spatstat; the integer outputs have no value here."""
    X, T, D = _cloud(case, seed)
    P, n, ks = X.double(), X.shape[0], _ks(case)
    nb = _bins(case)[2]
    e = torch.arange(nb + 1, dtype=torch.float64, device=X.device) * case["step"]
    edges = (e * e).float().double()
    outs = []
    for name in case["combos"].split("+"):
        ctr, nbr = COMBOS[name]
        ci = torch.nonzero(_in_set(T, ctr) & (D >= case["dsrf"])).flatten()
        ni = torch.nonzero(_in_set(T, nbr)).flatten()
        N = P[ni]
        hist = torch.zeros(nb, dtype=torch.float64, device=X.device)
        kth = torch.full((len(ks), n), float("nan"), dtype=torch.float64, device=X.device)
        for a in range(0, ci.numel(), 512):
            c = ci[a:a + 512]
            d2 = _d2_rows(P[c], N)
            d2.masked_fill_(c[:, None] == ni[None, :], float("inf"))
            d2.masked_fill_(d2 >= edges[-1], float("inf"))
            if case["gr"] and case["rdf"]:
                v = d2[torch.isfinite(d2)]
                b = torch.bucketize(v, edges, right=True) - 1
                hist += torch.bincount(b.clamp(0, nb - 1), minlength=nb).double()
            if case["per_central"] and ks:
                near = torch.full((c.numel(), max(ks)), float("inf"), dtype=torch.float64, device=X.device)
                m = min(max(ks), ni.numel())
                if m:
                    near[:, :m] = torch.topk(d2, m, dim=1, largest=False, sorted=True).values
                for q, k in enumerate(ks):
                    kth[q, c] = near[:, k - 1]
        out = {"rdf": None, "knn": None, "meta": None}
        if case["per_central"]:
            out["kth_d2"], out["n_within"] = kth if ks else None, None
        if case["gr"] and case["rdf"]:
            shell = 4.0 / 3.0 * math.pi * (e[1:] ** 3 - e[:-1] ** 3)
            norm = ci.numel() * (ni.numel() / _volume(case["cloud"], case["n"])) * shell
            out["g"] = hist / norm if ci.numel() * ni.numel() else hist
        outs.append(out)
    return outs


def _exact_soft(case, seed):
    """Smoothed RDF, gradient of the positions and of the scale."""
    s = prepare(dict(case, form="handle"), seed)
    X, D = s["X"], s["D"]
    P, n = X.double(), X.shape[0]
    nb, dr, sg = _bins(case)[2], case["step"], SOFT_SIGMA
    rc = case["stop"] + 6.0 * sg
    half = int(math.ceil(9.0 * sg / dr))
    off = torch.arange(-half, half + 1, device=X.device)
    ci = torch.nonzero(D >= case["dsrf"]).flatten()
    phi = torch.zeros(nb + 1, dtype=torch.float64, device=X.device)  # sum over the pairs of Phi((e - u)/sigma)

    def pairs():
        for a in range(0, ci.numel(), 512):
            c = ci[a:a + 512]
            d2 = _d2_rows(P[c], P)
            d2[torch.arange(c.numel(), device=X.device), c] = float("inf")
            r, j = torch.nonzero(d2 < rc * rc, as_tuple=True)
            yield c[r], j, d2[r, j].sqrt()

    for _, _, u in pairs():
        b = torch.round(u / dr).long()[:, None] + off[None, :]  # edges within reach; above them Phi = 1
        t = (b.double() * dr - u[:, None]) / sg
        val = 0.5 * torch.special.erfc(-t * math.sqrt(0.5))
        ok = (b >= 0) & (b <= nb)
        phi += torch.bincount(b[ok], weights=val[ok], minlength=nb + 1)
        above = torch.bincount((b[:, -1] + 1).clamp(0, nb + 1), minlength=nb + 2).double()
        phi += torch.cumsum(above, 0)[:nb + 1]
    h = phi[1:] - phi[:-1]
    f = s["factor"].double()
    G = 2.0 * (h * f - s["target"].double()) * f
    z = torch.zeros(1, dtype=torch.float64, device=X.device)
    coef = (torch.cat([G, z]) - torch.cat([z, G])) / sg  # W(u) = sum_e coef_e pdf((e - u)/sigma)
    grad = torch.zeros((n, 3), dtype=torch.float64, device=X.device)
    gs = torch.zeros(1, dtype=torch.float64, device=X.device)
    for i, j, u in pairs():
        b = torch.round(u / dr).long()[:, None] + off[None, :]
        t = (b.double() * dr - u[:, None]) / sg
        ok = ((b >= 0) & (b <= nb)).double()
        W = (coef[b.clamp(0, nb)] * ok * torch.exp(-0.5 * t * t)).sum(1) / math.sqrt(2.0 * math.pi)
        v = torch.where(u > 0, W / u, torch.zeros_like(u))[:, None] * (P[i] - P[j])
        grad.index_add_(0, i, v)
        grad.index_add_(0, j, -v)
        gs += (W * u).sum()
    return {"h": h, "grad": grad, "grad_scale": gs.reshape(1)}
