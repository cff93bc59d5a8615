"""The performance cases of this library: calls that a user of the (sub)halo search makes,
each through the public binding, from the smallest boxes to the 512^3 box.

Inputs are seeded mass-function boxes drawn on the GPU, of the same recipe as the
repository's generator: 40% of the particles in NFW hosts with dN/dM ~ M^-1.9 and
concentrations of 4 to 15, a tenth of each larger host's mass in Plummer subhalos, the rest
uniform. Two kinds of labels occur in earnest: those of the 3D FOF (hosts with their infall,
bridges and field groups), and pre-labelled hosts without a background, as a caller has them
who brings a catalogue of their own.

A case is {"call", "n", ...}: `call` names the entry point(s), `n` the particles.
"""
import math

import numpy as np
import torch

from paper_1902_01010_gb300 import vr

BOX = 1 << 21       # lattice points per axis
ALPHA = 1.9         # slope of the host mass function
NMIN, NSEARCH = 20, 160
NSE, NV = 256, 32   # the paper's N_se, N_v
FRAC = 0.4          # share of the particles in hosts


def listed():
    return [
        # 3D FOF. The 32^3 box is the smallest in use: launches and latency only. 256^3 is
        # the paper-scale test box; 512^3 the snapshot the paper analyses, and the largest.
        {"name": "fof3d 32^3", "call": "fof3d", "n": 32 ** 3},
        {"name": "fof3d 256^3", "call": "fof3d", "n": 256 ** 3},
        {"name": "fof3d 512^3", "call": "fof3d", "n": 512 ** 3},
        # Local velocity density on FOF halos: a box of no round size, with a bounded set of
        # halos, and the 256^3 box, whose halos run from 20 to several 100,000 members.
        {"name": "velden 1M", "call": "velden", "n": 999_983, "nse": NSE, "nv": NV},
        {"name": "velden 256^3", "call": "velden", "n": 256 ** 3, "nse": NSE, "nv": NV},
        # The same on a catalogue of the caller's own with smaller neighbour sets (the
        # faster, noisier setting), halos of up to two million members.
        {"name": "velden catalogue", "call": "velden catalogue", "n": 6_000_011, "nse": 64, "nv": 16},
        # Background cells, R and its fit, on an f_l that the caller already has.
        {"name": "outlier_ratio 200^3", "call": "outlier_ratio", "n": 200 ** 3},
        # Outlier linking alone: a caller who scans linking lengths or thresholds.
        {"name": "fof6d catalogue", "call": "fof6d catalogue", "n": 10_000_019},
        # Field 6DFOF of every FOF halo: all members are candidates.
        {"name": "fof6d_field 200^3", "call": "fof6d_field", "n": 200 ** 3},
        # Core search, cleaning and growth.
        {"name": "core_grow 128^3", "call": "core_grow", "n": 128 ** 3},
        # The whole search on the smallest box, and on a mid-sized one followed by the
        # two-stage linking and the significance cleaning.
        {"name": "search 32^3", "call": "search", "n": 32 ** 3},
        {"name": "search+grow+clean 80^3", "call": "search+grow+clean", "n": 80 ** 3},
    ]


# particles of each call's cases
RANGES = {
    "fof3d": (32 ** 3, 400 ** 3),
    "velden": (48 ** 3, 220 ** 3),
    "velden catalogue": (200_000, 5_000_000),
    "outlier_ratio": (48 ** 3, 190 ** 3),
    "fof6d catalogue": (200_000, 10_000_000),
    "fof6d_field": (48 ** 3, 190 ** 3),
    "core_grow": (32 ** 3, 120 ** 3),
    "search": (32 ** 3, 80 ** 3),
    "search+grow+clean": (32 ** 3, 76 ** 3),
}


def draw(rng):
    call = rng.choice(sorted(RANGES))
    lo, hi = RANGES[call]
    n = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    if rng.random() < 0.3:
        n = round(n ** (1.0 / 3.0)) ** 3  # a grid of particles, as simulations have
    case = {"call": call, "n": min(max(n, lo), hi)}
    if call.startswith("velden"):
        nse = rng.choice([64, 100, 256, 256, 512])
        case["nse"], case["nv"] = nse, min(rng.choice([16, 32, 32, 48]), nse)
    if call == "fof3d":
        case["link_num"], case["link_den"] = rng.choice([(1, 5), (1, 5), (4, 25), (7, 25)])
    return case


# ------------------------------------------------------------------------------ inputs
def mean_spacing(n):
    return BOX / n ** (1.0 / 3.0)


def link_d2(n, num=1, den=5):
    """Smallest integer T with d^2 < T <=> d < (num/den) of the mean spacing."""
    return int(math.floor((num / den * mean_spacing(n)) ** 2)) + 1


def _power(rs, size, lo, hi):
    e = 1.0 - ALPHA
    return (lo ** e + rs.random_sample(size) * (hi ** e - lo ** e)) ** (1.0 / e)


def _isotropic(rs, size):
    d = rs.standard_normal((size, 3))
    return d / np.linalg.norm(d, axis=1, keepdims=True)


def _nfw_m(x):
    return np.log1p(x) - x / (1.0 + x)


def _hosts(n, rs, catalogue):
    """Blob table (numpy): one row per host's smooth part and per subhalo."""
    hi = min(4e6, n / 3.0) if catalogue else min(1e6, n / 16.0)
    total = n if catalogue else int(FRAC * n)
    sizes = np.zeros(0, np.int64)
    while sizes.sum() < total:
        sizes = np.concatenate([sizes, np.rint(_power(rs, max(64, total // 300), 20.0, hi)).astype(np.int64)])
    sizes = sizes[:int(np.searchsorted(np.cumsum(sizes), total)) + 1]
    over = int(sizes.sum()) - total  # the last host takes what is left
    sizes[-1] -= over
    if sizes[-1] < NMIN:
        sizes[0] += sizes[-1]
        sizes = sizes[:-1]
    nh = len(sizes)
    nbar = n / float(BOX) ** 3
    r200 = lambda m: np.cbrt(3.0 * m / (4.0 * math.pi * 200.0 * nbar))  # noqa: E731
    conc = rs.uniform(4.0, 15.0, nh)
    sigma = 100.0 * np.cbrt(sizes / 1000.0)
    centre = rs.random_sample((nh, 3)) * BOX
    bulk = 30.0 * rs.standard_normal((nh, 3))
    # subhalos: power-law mass ratios, about a tenth of the mass of hosts of 200 and more
    parent = np.repeat(np.arange(nh), np.where(sizes >= 200, 19, 0))
    m = np.rint(_power(rs, len(parent), 1e-3, 1e-1) * sizes[parent]).astype(np.int64)
    before = np.cumsum(m) - m
    first = np.searchsorted(parent, parent)
    keep = (m >= NMIN) & (before - before[first] + m <= 0.2 * sizes[parent])
    parent, m = parent[keep], m[keep]
    # a subhalo sits at a radius drawn from its host's profile
    lo, up = np.zeros(len(m)), conc[parent].copy()
    want = rs.random_sample(len(m)) * _nfw_m(conc[parent])
    for _ in range(40):
        mid = 0.5 * (lo + up)
        low = _nfw_m(mid) < want
        lo, up = np.where(low, mid, lo), np.where(low, up, mid)
    place = centre[parent] + (lo * r200(sizes[parent]) / conc[parent])[:, None] * _isotropic(rs, len(m))
    smooth = sizes.copy()
    np.subtract.at(smooth, parent, m)
    return dict(
        count=np.concatenate([smooth, m]),
        centre=np.concatenate([centre, place]),
        scale=np.concatenate([r200(sizes) / conc, r200(m) / 5.0]),
        conc=np.concatenate([conc, np.zeros(len(m))]),  # 0: Plummer
        bulk=np.concatenate([bulk, bulk[parent] + sigma[parent, None] * rs.standard_normal((len(m), 3))]),
        sigma=np.concatenate([sigma, sigma[parent] * np.cbrt(m / sizes[parent])]),
        host=np.concatenate([np.arange(nh), parent]),
        sub=np.concatenate([np.zeros(nh, bool), np.ones(len(m), bool)]),
        sizes=sizes, host_sigma=sigma)


def particles(n, seed, catalogue=False):
    """Positions int32 [n, 3] and velocities float32 [n, 3] on the GPU, the host of each
    particle (int32, -1: background), whether it lies in a subhalo, and the host table."""
    dev = torch.device("cuda")
    g = torch.Generator(device=dev).manual_seed(seed)
    b = _hosts(n, np.random.RandomState((seed * 7919 + n) % (1 << 32)), catalogue)
    up = lambda x: torch.from_numpy(np.ascontiguousarray(x)).to(dev)  # noqa: E731
    count = up(b["count"])
    blob = torch.repeat_interleave(torch.arange(len(b["count"]), device=dev), count)
    nin = blob.numel()
    conc = up(b["conc"].astype(np.float32))[blob]
    u = torch.rand(nin, device=dev, generator=g)
    # NFW radius in units of r_s by bisection, Plummer radius truncated at 10 a
    want = u * (torch.log1p(conc) - conc / (1.0 + conc))
    lo, hi = torch.zeros_like(conc), conc.clone()
    for _ in range(22):
        mid = 0.5 * (lo + hi)
        low = (torch.log1p(mid) - mid / (1.0 + mid)) < want
        lo, hi = torch.where(low, mid, lo), torch.where(low, hi, mid)
    plummer = torch.rsqrt((u * 0.985).clamp_min(1e-9).pow(-2.0 / 3.0) - 1.0)
    r = torch.where(conc > 0, lo, plummer) * up(b["scale"].astype(np.float32))[blob]
    del u, want, lo, hi, mid, low, plummer, conc
    d = torch.randn(nin, 3, device=dev, generator=g)
    d *= (r / d.norm(dim=1).clamp_min(1e-20))[:, None]
    pos = torch.empty(n, 3, dtype=torch.int32, device=dev)
    pos[nin:] = torch.randint(0, BOX, (n - nin, 3), device=dev, generator=g, dtype=torch.int32)
    centre = up(np.floor(b["centre"]).astype(np.int32))
    for a in range(3):
        pos[:nin, a] = centre[:, a][blob] + torch.floor(d[:, a]).to(torch.int32)
    pos &= BOX - 1
    del d, r
    vel = torch.randn(n, 3, device=dev, generator=g)
    sigma, bulk = up(b["sigma"].astype(np.float32)), up(b["bulk"].astype(np.float32))
    vel[:nin] *= sigma[blob][:, None]
    vel[:nin] += bulk[blob]
    vel[nin:] *= 30.0
    host = torch.full((n,), -1, dtype=torch.int32, device=dev)
    host[:nin] = up(b["host"].astype(np.int32))[blob]
    sub = torch.zeros(n, dtype=torch.bool, device=dev)
    sub[:nin] = up(b["sub"])[blob]
    del blob
    mix = torch.randperm(n, device=dev, generator=g)  # particles come in no order
    return pos[mix], vel[mix], host[mix], sub[mix], b


def catalogue_labels(host, nhost):
    """Minimum particle index of each particle's host: the form of the 3D FOF labels."""
    n = host.numel()
    first = torch.full((nhost,), n, dtype=torch.int32, device=host.device)
    idx = torch.arange(n, dtype=torch.int32, device=host.device)
    first.scatter_reduce_(0, host.long(), idx, "amin")
    return first[host.long()], first


def prepare(case, seed):
    call, n = case["call"], case["n"]
    catalogue = call.endswith("catalogue")
    pos, vel, host, sub, b = particles(n, seed, catalogue)
    ctx = vr.Context(torch.cuda.current_device())
    ctx.workspace(n, vr.Params.default())
    s = dict(case, ctx=ctx, pos=pos, d2=link_d2(n, case.get("link_num", 1), case.get("link_den", 5)),
             lx=0.2 * mean_spacing(n), lx_sub=0.1 * mean_spacing(n))
    if call == "fof3d":
        return s
    s["vel"] = vel
    # the caller's halo table, as long as the calls may need it; rows behind the last halo
    # keep what they hold
    s["table"] = torch.zeros(n // NMIN + 1, vr.HALO_COLS, dtype=torch.float64, device=pos.device)
    if call.startswith("search"):
        return s
    s["params"] = vr.Params.default(**{k: case[k] for k in ("nse", "nv") if k in case})
    ctx.workspace(n, s["params"])
    if not catalogue:
        s["label"] = ctx.fof3d(pos, s["d2"])
        ctx.sync()
    else:
        s["label"], first = catalogue_labels(host, len(b["sizes"]))
    g = torch.Generator(device=pos.device).manual_seed(seed + 1)
    if call == "outlier_ratio":
        # the Maxwellian density of the host's dispersion, with the scatter of N_v = 32
        # neighbours and the excess of cold subhalos
        sig = torch.full((n,), 60.0, device=pos.device)
        m = host >= 0
        sig[m] = torch.from_numpy(b["host_sigma"].astype(np.float32)).to(pos.device)[host[m].long()]
        lnf = -1.5 * torch.log(2.0 * math.pi * sig * sig) - 0.5 * (vel / sig[:, None]).square().sum(1).clamp(max=30.0)
        lnf += 0.3 * torch.randn(n, device=pos.device, generator=g)
        lnf += sub.float() * (1.0 + torch.rand(n, device=pos.device, generator=g))
        s["f_l"] = torch.exp(lnf)
    if call == "fof6d catalogue":
        # outliers: the subhalo members, and the tail of the smooth ones
        ell = torch.randn(n, device=pos.device, generator=g)
        s["ell"] = torch.where(sub, 3.5 + 1.2 * ell, ell)
        order = torch.argsort(first)  # rows in label order
        sizes = torch.from_numpy(b["sizes"]).to(pos.device)[order]
        sigma = torch.from_numpy(b["host_sigma"]).to(pos.device)[order]
        bulk = torch.from_numpy(np.ascontiguousarray(b["bulk"][:len(b["sizes"])])).to(pos.device)[order]
        rows = torch.zeros(len(sizes), vr.HALO_COLS, dtype=torch.float64, device=pos.device)
        rows[:, vr.H_LABEL], rows[:, vr.H_NH] = first[order].double(), sizes.double()
        rows[:, vr.H_SEARCHED] = (sizes >= NSEARCH).double()
        rows[:, vr.H_VFX:vr.H_VFZ + 1] = bulk
        rows[:, vr.H_SIGMA], rows[:, vr.H_LX2], rows[:, vr.H_LV2] = sigma, s["lx_sub"] ** 2, sigma ** 2
        s["rows"] = rows[sizes >= NMIN].contiguous()
    return s


# --------------------------------------------------------------------------------- run
def run(s):
    ctx, call = s["ctx"], s["call"]
    if call == "fof3d":
        return ctx.fof3d(s["pos"], s["d2"])
    if call.startswith("velden"):
        return ctx.velden(s["pos"], s["vel"], s["label"], s["params"])
    if call == "outlier_ratio":
        R, ell, halos = ctx.outlier_ratio(s["pos"], s["vel"], s["f_l"], s["label"], s["params"])
        s["table"][:halos.shape[0]] = halos
        return {"R": R, "ell": ell, "halos": s["table"]}
    if call == "fof6d catalogue":
        return ctx.fof6d(s["pos"], s["vel"], s["ell"], s["label"], s["rows"], s["params"])
    if call == "fof6d_field":
        label6, rows = ctx.fof6d_field(s["pos"], s["vel"], s["label"], s["lx"], 1.25, s["params"],
                                       halos=s["table"])
        return {"label6": label6, "halos": s["table"], "nhalo": rows.shape[0]}
    new = lambda dtype: torch.empty(s["n"], dtype=dtype, device=s["pos"].device)  # noqa: E731
    if call == "core_grow":
        out = dict({k: new(torch.int32) for k in ("core", "level", "grown")}, halos=s["table"])
        return ctx.core_grow(s["pos"], s["vel"], s["label"], None, s["lx"], 1.25, s["params"], out=out)
    # the whole search of a box
    label = ctx.fof3d(s["pos"], s["d2"])
    out = dict({k: new(torch.float32) for k in ("f_l", "R", "ell")}, label6=new(torch.int32),
               halos=s["table"])
    out = ctx.find_substructure(s["pos"], s["vel"], label, s["lx_sub"], 1.0, out=out)
    out["label"] = label
    if call == "search+grow+clean":
        ctx.grow_groups(s["pos"], s["vel"], out["ell"], label, out["halos"][:out["nhalo"]], out["label6"])
        out["ngroups"] = ctx.clean_groups(out["ell"], out["label6"])
    return out


def work(case):
    """Bytes and 32-bit operations of one pass that the method cannot do without.

    3D FOF: positions in, labels out (16 B), and the 13 half-neighbour cells' pair test of
    8 operations per particle. f_l: 28 B in and 4 B out; per member of a larger halo N_se
    position and N_se velocity distances of 8 operations, a selection of 1 per element and
    an N_v-term sum of 3. Cells and R: positions, velocities, labels and f_l in, R and ell
    out, seven cells' interpolation of about 200 operations. Links: positions, velocities,
    labels and ell in, labels out. The share of particles in halos is the generator's.
    """
    call, n = case["call"], case["n"]
    halo = 1.0 if call.endswith("catalogue") else FRAC
    nse, nv = case.get("nse", NSE), case.get("nv", NV)
    fof = {"bytes": 16.0 * n, "flops": 13 * 8.0 * n}
    fl = {"bytes": 32.0 * n, "flops": halo * n * (18.0 * nse + 3.0 * nv)}
    ratio = {"bytes": 40.0 * n, "flops": halo * n * 200.0}
    links = {"bytes": 36.0 * n, "flops": halo * n * 40.0}
    parts = {"fof3d": [fof], "velden": [fl], "outlier_ratio": [ratio], "fof6d": [links],
             "fof6d_field": [links], "core_grow": [links, ratio], "search": [fof, fl, ratio, links],
             "search+grow+clean": [fof, fl, ratio, links, links]}[call.split(" ")[0]]
    return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}


# ------------------------------------------------------------------------------- exact
# Plain 64-bit restatements for the calls whose outputs are computed numbers, on boxes where
# they end in seconds. Labels are whole numbers; ell and the fit's columns come from an
# iterative minimiser whose end point is fixed only to about the square root of its stopping
# rule, so they have no value here.
EXACT_PAIRS = 3e10   # member pairs of all halos, brute force
EXACT_MEMBERS = 150_000  # members of searched halos, host-side trees


def _halos(label, nmin):
    """Members (ascending index) of each group of at least nmin, in label order."""
    lab = label.cpu().numpy().astype(np.int64)
    order = np.argsort(lab, kind="stable")
    ids, start, size = np.unique(lab[order], return_index=True, return_counts=True)
    return [order[a:a + c] for i, a, c in zip(ids, start, size) if c >= nmin]


def _unwrap(pos, m):
    p = pos[m].astype(np.int64)
    d = p - p[0]
    d = np.where(d >= BOX // 2, d - BOX, np.where(d < -(BOX // 2), d + BOX, d))
    return p[0] + d


def _exact_velden(pos, vel, halos, n, nse, nv):
    """Brute force on the GPU: exact integer keys, FP64 kernel sums."""
    out = np.full(n, np.nan)
    for m in halos:
        x = torch.from_numpy(_unwrap(pos, m)).cuda()
        v = torch.from_numpy(vel[m].astype(np.float64)).cuda()
        k, got = min(nse, len(m)), []
        rank = torch.arange(len(m), device="cuda")
        step = max(1, int(3e8) // len(m))
        for a in range(0, len(m), step):
            q = x[a:a + step]
            key = (q[:, None, 0] - x[None, :, 0]).square_()
            for c in (1, 2):
                key += (q[:, None, c] - x[None, :, c]).square_()
            key = (key << 22) + rank
            near = torch.topk(key, k, dim=1, largest=False, sorted=False).values & ((1 << 22) - 1)
            del key
            d2 = (v[near] - v[a:a + step][:, None]).square().sum(2)
            h2 = torch.topk(d2, min(nv, k), dim=1, largest=False).values[:, -1:]
            w = torch.where(d2 < h2, 1.0 - d2 / h2, 0.0).sum(1)
            f = 15.0 / (8.0 * math.pi) / h2[:, 0].pow(1.5) * w / k
            got.append(torch.where(h2[:, 0] > 0, f, math.inf))
        out[m] = torch.cat(got).cpu().numpy()
    return out


def _split(x, beg, ncell, lo, hi, tree):
    """Entropy kd-tree of the members `beg`; returns the node number."""
    me = len(tree)
    tree.append(None)
    n = len(beg)
    if n > ncell:
        p = x[beg]
        nb = int(round(n ** (1.0 / 3.0)))
        nb -= nb ** 3 > n
        nb = max(2, nb + ((nb + 1) ** 3 <= n))
        mn, mx = p.min(0), p.max(0)
        S = np.full(3, -1.0)
        for a in range(3):
            if mx[a] > mn[a]:
                f = np.bincount((p[:, a] - mn[a]) * nb // (mx[a] - mn[a] + 1)) / n
                f = f[f > 0]
                S[a] = -(f * np.log(f)).sum() / math.log(nb)
        left = [a for a in range(3) if mx[a] > mn[a]]
        while left:
            a = left[0]
            for c in left[1:]:
                if S[c] > S[a] + 1e-12:
                    a = c
            left.remove(a)
            xs = int(np.partition(p[:, a], n // 2)[n // 2])
            isl = p[:, a] < xs
            if not isl.any():
                continue
            hl, lr = hi.copy(), lo.copy()
            hl[a], lr[a] = xs, xs
            tree[me] = (a, xs, _split(x, beg[isl], ncell, lo, hl, tree), _split(x, beg[~isl], ncell, lr, hi, tree))
            return me
    tree[me] = (-1, beg, lo, hi)
    return me


def _locate(tree, p):
    """Node of the leaf that holds each point of p."""
    at, todo = np.zeros(len(p), np.int64), [(0, np.arange(len(p)))]
    while todo:
        k, idx = todo.pop()
        a = tree[k][0]
        if a < 0:
            at[idx] = k
            continue
        isl = p[idx, a] < tree[k][1]
        todo += [(tree[k][2], idx[isl]), (tree[k][3], idx[~isl])]
    return at


def _exact_ratio(pos, vel, f_l, halos, n):
    out = np.full(n, np.nan)
    for m in halos:
        if len(m) < NSEARCH:
            continue
        x, v = _unwrap(pos, m), vel[m].astype(np.float64)
        ncell = int(0.01 * len(m))
        ncell = ncell if ncell >= 100 else min(100, len(m) // 8)
        tree = []
        rlo, rhi = x.min(0), x.max(0) + 1
        _split(x, np.arange(len(m)), ncell, rlo, rhi, tree)
        xm, vm, sg, lo, hi = (np.zeros((len(tree),) + k) for k in ((3,), (3,), (3, 3), (3,), (3,)))
        own = np.zeros(len(m), np.int64)
        for k, node in enumerate(tree):
            if node[0] < 0:
                xm[k], vm[k] = x[node[1]].mean(0), v[node[1]].mean(0)
                d = v[node[1]] - vm[k]
                sg[k] = d.T @ d / len(node[1])
                lo[k], hi[k] = node[2], node[3]
                own[node[1]] = k
        cells, use = [own], [np.ones(len(m), bool)]
        for a in range(3):
            for edge in (lo[own, a] - 1, hi[own, a]):
                p = x.copy()
                p[:, a] = edge
                c = _locate(tree, p)
                ok = (p[:, a] >= rlo[a]) & (p[:, a] < rhi[a])
                for k, w in zip(cells, use):
                    ok &= ~(w & (k == c))
                cells.append(c)
                use.append(ok)
        cells, use = np.array(cells), np.array(use)
        d = np.linalg.norm(x[None] - xm[cells], axis=2)
        with np.errstate(divide="ignore", invalid="ignore"):
            w = np.where(use, 1.0 / d, 0.0)
        zero = (use & (d == 0)).any(0)
        w[:, zero] = (use & (d == 0))[:, zero]
        w /= w.sum(0)
        vb, S = np.einsum("km,kma->ma", w, vm[cells]), np.einsum("km,kmab->mab", w, sg[cells])
        dv = v - vb
        q = np.einsum("ma,ma->m", dv, np.linalg.solve(S, dv[..., None])[..., 0])
        ln_bg = -0.5 * q - 1.5 * math.log(2.0 * math.pi) - 0.5 * np.linalg.slogdet(S)[1]
        out[m] = np.log(f_l[m].astype(np.float64)) - ln_bg
    return out


def exact(case, seed):
    call, n = case["call"], case["n"]
    if call.startswith(("fof", "core")):
        return None
    s = prepare(case, seed)
    if call.startswith("search"):
        return None if n > 40 ** 3 else _exact_search(s, n)
    halos = _halos(s["label"], NMIN)
    pos, vel = s["pos"].cpu().numpy(), s["vel"].cpu().numpy()
    if call.startswith("velden"):
        if sum(float(len(m)) ** 2 for m in halos) > EXACT_PAIRS:
            return None
        return _exact_velden(pos, vel, halos, n, case["nse"], case["nv"])
    if sum(len(m) for m in halos if len(m) >= NSEARCH) > EXACT_MEMBERS:
        return None
    return {"R": _exact_ratio(pos, vel, s["f_l"].cpu().numpy(), halos, n), "ell": None, "halos": None}


def _exact_search(s, n):
    """f_l and R of a small box; its 3D groups by brute force over the GPU."""
    x = s["pos"].long()
    label = torch.arange(n, device=x.device)
    pairs = []
    for a in range(0, n, 2048):
        d = (x[a:a + 2048, None] - x[None]).abs_()
        d = torch.minimum(d, BOX - d).square_().sum(2)
        i, j = torch.nonzero(d < s["d2"], as_tuple=True)
        pairs.append(torch.stack([i + a, j]))
    i, j = torch.cat(pairs, 1)
    while True:  # minimum label over links until nothing changes
        new = label.scatter_reduce(0, i, label[j], "amin")
        new = new[new]
        if torch.equal(new, label):
            break
        label = new
    halos = _halos(label, NMIN)
    pos, vel = s["pos"].cpu().numpy(), s["vel"].cpu().numpy()
    f_l = _exact_velden(pos, vel, halos, n, NSE, NV)
    R = _exact_ratio(pos, vel, f_l, halos, n)
    out = {k: None for k in ("ell", "halos", "label", "label6", "nhalo")}
    return dict(out, f_l=f_l, R=R, **({"ngroups": None} if s["call"] != "search" else {}))
