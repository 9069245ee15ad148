"""The calls whose speed is measured: what a simulation program asks of this
library, through its public entry points, from one thousand particles to two
million.

Kinds of pass (`case["kind"]`):
  list      build and query, and the neighbour matrix padded with -1 past each
            row's end, as a program that keeps the list for its own kernels
            takes it (FP32 or double-precision particle data);
  step      one molecular-dynamics step that rebuilds its Verlet list: build,
            traversal, per-particle energies and forces (liquid, liquid/vapor
            or size-asymmetric mixture);
  forces    one step between two rebuilds: energies and forces over the list of
            the last rebuild, at positions that have moved within the skin;
  train     forward and backward of the differentiable energy over a batch of
            two-type systems, the list rebuilt for the positions of the step;
  ensemble  many independent systems of uneven size through one captured
            launch sequence, then their energies and forces.

Positions are jittered lattices (the liquids), random-wave liquid/vapor
domains, or lattices around large spheres; units are those of the
Lennard-Jones potential.  Options are the library's defaults, or the subtree
size of 64 leaves that the autotuner settles on for large systems.
"""
import math

import numpy as np
import torch

from paper_1901_08088_gb300 import _lib
from paper_1901_08088_gb300.batch import BatchedNeighborList
from paper_1901_08088_gb300.lj import lj_energy, pack_positions
from paper_1901_08088_gb300.qbvh import NeighborList, check, qbvh_lj_forward

WCA = 2.0 ** (1.0 / 6.0)   # cutoff of the purely repulsive potential


# ------------------------------------------------------------------- cases

def _case(kind, **kw):
    c = dict(kind=kind, n=4096, n_sys=1, rho=0.8, jitter=0.25, r_cut=3.0, skin=0.3, shape="liquid", data="f32",
             bundle=0, node_format=0, one_tree=False)
    c.update(kw)
    return c


def listed():
    return [
        # a small molecule's box rebuilt every few steps: launches and latency
        _case("list", name="list_n1000", n=1000, rho=0.6, jitter=0.3, skin=0.4),
        # the plain build + query of one small fluid
        _case("list", name="list_n4096", n=4096, rho=0.6, jitter=0.3, skin=0.4),
        # an ordinary single-GPU simulation with library defaults, N not a multiple of anything
        _case("step", name="step_n30011", n=30011, rho=0.7),
        # repulsive (WCA) fluid: short cutoff, few neighbours
        _case("step", name="step_wca_n131072", n=131072, rho=0.8, r_cut=WCA, skin=0.3),
        # double-precision particle data of a mid-size fluid
        _case("list", name="list_f64_n131072", n=131072, rho=0.8, data="f64", bundle=64),
        # steps between rebuilds: forces over a list that is kept
        _case("forces", name="forces_n262144", n=262144, rho=0.8),
        # large colloids in a solvent: one tree and one radius per type pair
        _case("step", name="step_mixture_L100", n=395280, rho=0.5, shape="mixture", skin=0.4),
        # liquid/vapor coexistence: uneven density, a third of the box nearly empty
        _case("step", name="step_vapor_n1000000", n=1000000, rho=0.2, shape="vapor", skin=0.0, bundle=64),
        # potential fitting: energies, forces and parameter gradients of a batch of two-type systems
        _case("train", name="train_32x65536", n=65536, n_sys=32, jitter=0.3, r_cut=2.5, bundle=64, one_tree=True),
        # hundreds of independent systems of uneven size
        _case("ensemble", name="ensemble_256", n=50000, n_sys=256, rho=0.6, jitter=0.3, r_cut=2.5, bundle=64),
        # the large production fluid, tuned options
        _case("step", name="step_n2097152", n=2097152, rho=0.8, bundle=64),
    ]


def draw(rng):
    def logn(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["list", "list", "step", "step", "step", "forces", "train", "ensemble"])
    c = dict(rho=round(rng.uniform(0.3, 0.9), 3), jitter=round(rng.uniform(0.2, 0.3), 3),
             r_cut=rng.choice([WCA, 2.5, 3.0, 3.0]), skin=rng.choice([0.3, 0.4]), bundle=rng.choice([0, 64]))
    if kind == "list":
        c.update(n=logn(1000, 262144), data=rng.choice(["f32", "f32", "f64"]), node_format=rng.choice([0, 0, 1]))
    elif kind == "step":
        shape = rng.choice(["liquid", "liquid", "liquid", "vapor", "mixture"])
        if shape == "liquid":
            c.update(n=logn(1000, 1500000), node_format=rng.choice([0, 0, 1]))
        elif shape == "vapor":
            c.update(n=logn(100000, 1000000), rho=0.2, r_cut=3.0)
        else:
            c.update(n=logn(40000, 395280), rho=0.5, r_cut=3.0)
        c["shape"] = shape
    elif kind == "forces":
        c.update(n=logn(1000, 1500000))
    elif kind == "train":
        n = logn(1000, 65536)
        c.update(n=n, n_sys=max(1, min(32, logn(1, 32), 1500000 // n)), r_cut=2.5, one_tree=rng.choice([True, False]))
    else:
        c.update(n=logn(2000, 50000), n_sys=logn(4, 256), r_cut=2.5)
    return _case(kind, **c)


# ------------------------------------------------------------------- inputs

def _edge(n, rho):
    return float(np.float32((n / rho) ** (1.0 / 3.0)))


def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _lattice(n, L, jitter, g):
    """n of the m^3 sites of a simple-cubic lattice, each moved by up to `jitter` per axis."""
    m = int(round(n ** (1.0 / 3.0)))
    m += m ** 3 < n
    sites = torch.arange(m ** 3, device="cuda")
    if m ** 3 > n:
        sites = torch.randperm(m ** 3, generator=g, device="cuda")[:n].sort().values
    ijk = torch.stack([sites // (m * m), (sites // m) % m, sites % m], 1).double()
    return (ijk + 0.5) * (L / m) + jitter * (2 * torch.rand((n, 3), generator=g, device="cuda", dtype=torch.float64) - 1)


def _wrap32(x, L):
    x = torch.remainder(x, L).float()
    return torch.where((x >= L) | (x < 0), torch.zeros_like(x), x)


def _vapor(n, rho, jitter, g):
    """Liquid/vapor domains: a random-wave field thresholded to the lever rule, a
    lattice at liquid density where it is high, a sparse lattice elsewhere."""
    L, liquid, vapor = _edge(n, rho), 0.72, 0.02
    k = torch.randn((64, 3), generator=g, device="cuda", dtype=torch.float64)
    k = k / k.norm(dim=1, keepdim=True) * (2 * math.pi / 20.0)
    k = torch.round(k * L / (2 * math.pi)) * (2 * math.pi / L)
    phase = 2 * math.pi * torch.rand(64, generator=g, device="cuda", dtype=torch.float64)

    def field(x):
        return sum(torch.cos(x @ k[i:i + 16].T + phase[i:i + 16]).sum(1) for i in range(0, 64, 16))

    def grid(density):
        m = int(math.ceil((density * L ** 3) ** (1.0 / 3.0)))
        a = (torch.arange(m, device="cuda", dtype=torch.float64) + 0.5) * (L / m)
        x = torch.stack(torch.meshgrid(a, a, a, indexing="ij"), -1).reshape(-1, 3)
        return x, L / m

    xl, al = grid(liquid)
    f = field(xl)
    # the threshold that leaves the liquid its share of the n particles, kept within the sites there are
    n_vap_sites = int(round(vapor * L ** 3 * (1 - (rho - vapor) / (liquid - vapor))))
    keep = f.topk(n - n_vap_sites).indices.sort().values
    xl = xl[keep] + jitter * (2 * torch.rand((keep.numel(), 3), generator=g, device="cuda", dtype=torch.float64) - 1)
    xv, av = grid(1.3 * vapor)
    low = (-field(xv)).topk(n_vap_sites).indices.sort().values
    xv = xv[low] + 0.2 * av * (2 * torch.rand((n_vap_sites, 3), generator=g, device="cuda", dtype=torch.float64) - 1)
    x = torch.cat([xl, xv])
    return x[torch.randperm(n, generator=g, device="cuda")], L


def _mixture(n_small, rho, jitter, seed, g):
    """Spheres of diameter 10 by random sequential addition, small particles on a
    jittered lattice outside their cores; the large ones come last."""
    n_large = max(4, int(round(n_small * 400 / 395280)))
    L = float(np.float32((n_small / rho + n_large * 4.0 / 3.0 * math.pi * 125) ** (1.0 / 3.0)))
    r = np.random.default_rng(seed)
    c = np.empty((0, 3))
    while len(c) < n_large:
        p = r.uniform(0, L, 3)
        d = c - p
        d -= L * np.rint(d / L)
        if not len(c) or (d * d).sum(1).min() >= 100.0:
            c = np.vstack([c, p])
    ct = torch.from_numpy(c).cuda()
    m = int(math.ceil((1.06 * n_small / (1 - n_large * 4.0 / 3.0 * math.pi * 125 / L ** 3)) ** (1.0 / 3.0)))
    x = _lattice(m ** 3, L, min(jitter, 0.25 * L / m), g)
    far = torch.ones(len(x), dtype=torch.bool, device="cuda")
    for p in ct:
        d = x - p
        d -= L * torch.round(d / L)
        far &= (d * d).sum(1) >= 25.0
    x = x[far]
    x = x[torch.randperm(len(x), generator=g, device="cuda")[:n_small].sort().values]
    types = torch.cat([torch.zeros(len(x), dtype=torch.int32), torch.ones(n_large, dtype=torch.int32)]).cuda()
    return torch.cat([x, ct]), types, L


def _matrices(case):
    """list radii, cutoffs, eps and sigma of every type pair."""
    if case["shape"] == "mixture":   # large pairs repel only, from their diameters
        rc = np.array([[case["r_cut"], 5.5], [5.5, 10.0]], np.float32)
        return rc + np.float32(case["skin"]), rc, np.ones((2, 2), np.float32), np.array([[1.0, 4.9], [4.9, 8.9]], np.float32)
    T = 2 if case["kind"] == "train" else 1
    rc = np.full((T, T), case["r_cut"], np.float32)
    eps = np.array([[1.0, 1.5], [1.5, 0.5]], np.float32)[:T, :T]
    sig = np.array([[1.0, 0.88], [0.88, 0.8]], np.float32)[:T, :T]
    return rc + np.float32(case["skin"]), rc, eps, sig


def _inputs(case, seed):
    """Positions [n, 3], types [n], system offsets and box edges."""
    g = _gen(seed)
    T = 2 if case["kind"] == "train" else 1
    if case["shape"] == "mixture":
        x, types, L = _mixture(case["n"], case["rho"], case["jitter"], seed, g)
        return _wrap32(x, L), types, [0, len(types)], [L]
    if case["shape"] == "vapor":
        x, L = _vapor(case["n"], case["rho"], case["jitter"], g)
        return _wrap32(x, L), torch.zeros(case["n"], dtype=torch.int32, device="cuda"), [0, case["n"]], [L]
    if case["data"] == "f64":
        L = (case["n"] / case["rho"]) ** (1.0 / 3.0)
        x = torch.remainder(_lattice(case["n"], L, case["jitter"], g), L)
        x = torch.where((x >= L) | (x < 0), torch.zeros_like(x), x)
        return x, torch.zeros(case["n"], dtype=torch.int32, device="cuda"), [0, case["n"]], [L]
    if case["kind"] == "ensemble":   # sizes spread evenly over their logarithm, densities uniform
        r = np.random.default_rng(seed)
        ns, rhos = _sizes(case), r.uniform(0.5 * case["rho"], 1.5 * case["rho"], case["n_sys"])
        r.shuffle(ns)
        rhos = np.minimum(rhos, 0.9)
    else:
        ns, rhos = [case["n"]] * case["n_sys"], [case["rho"]] * case["n_sys"]
    xs, off, Ls = [], [0], []
    for n, rho in zip(ns, rhos):
        L = _edge(int(n), float(rho))
        xs.append(_wrap32(_lattice(int(n), L, case["jitter"], g), L))
        off.append(off[-1] + int(n))
        Ls.append(L)
    types = torch.zeros(off[-1], dtype=torch.int32, device="cuda")
    if T == 2:
        for k in range(len(Ls)):
            types[off[k] + torch.randperm(off[k + 1] - off[k], generator=g, device="cuda")[: (off[k + 1] - off[k]) // 2]] = 1
    return torch.cat(xs), types, off, Ls


def _sizes(case):
    lo, hi = min(500, case["n"]), case["n"]
    t = (np.arange(case["n_sys"]) + 0.5) / case["n_sys"]
    return np.rint(lo * (hi / lo) ** t).astype(np.int64)


def _mean_neighbors(case, r):
    rho = {"vapor": 0.72, "mixture": case["rho"]}.get(case["shape"], case["rho"])
    return rho * 4.0 / 3.0 * math.pi * float(r) ** 3


def _cap(case, r_list):
    """Row capacity a program would reserve: the densest region's mean and a margin."""
    if case["shape"] == "mixture":
        return 320
    dens = 1.5 if case["kind"] == "ensemble" else 1.0
    return int(math.ceil((1.35 * dens * _mean_neighbors(case, r_list[0, 0]) + 24) / 32) * 32)


def _moved(x, L, skin, seed):
    g = _gen(seed + 1)
    d = (0.28 * skin) * (2 * torch.rand(x.shape, generator=g, device="cuda") - 1)   # under skin / 2
    return _wrap32(x.double() + d.double(), L)


def prepare(case, seed):
    r_list, r_cut, eps, sig = _matrices(case)
    x, types, off, Ls = _inputs(case, seed)
    n, S, T = x.shape[0], len(Ls), r_cut.shape[0]
    s = dict(kind=case["kind"], L=Ls[0], off=off, Ls=Ls, T=T, r_list=r_list, r_cut=r_cut, cap=_cap(case, r_list))
    opts = {}
    if case["bundle"]:
        opts[_lib.QBVH_OPT_BUNDLE] = case["bundle"]
    if case["node_format"]:
        opts[_lib.QBVH_OPT_NODE_FORMAT] = case["node_format"]
    if case["one_tree"]:
        opts[_lib.QBVH_OPT_TYPE_TREES] = 0
    s["eps"], s["sig"] = torch.from_numpy(eps.copy()).cuda(), torch.from_numpy(sig.copy()).cuda()
    if case["data"] == "f64":
        s["pos64"] = torch.cat([x, types.double()[:, None]], 1).contiguous()
    else:
        s["pos4"] = pack_positions(x, types)
    if case["kind"] == "ensemble":
        s["batch"] = BatchedNeighborList(s["pos4"], off, Ls, r_list, n_types=T, cap=s["cap"], options=opts)
        s["batch"].capture()
        s["nl"] = s["batch"].nl
    else:
        s["nl"] = NeighborList()
        for k, v in opts.items():
            s["nl"].set_option(k, v)
    if case["kind"] == "list":
        s["column"] = torch.arange((s["cap"] + 7) // 8 * 8, device="cuda", dtype=torch.int32)
    if case["kind"] == "train":
        s["xyz"], s["types"] = x.requires_grad_(), types
        s["eps"].requires_grad_()
        s["sig"].requires_grad_()
        s["weight"] = torch.linspace(0.5, 1.5, S, device="cuda", dtype=torch.float64)
    else:
        s["e"] = torch.empty(n, device="cuda")
        s["F"] = torch.empty((n, 3), device="cuda")
        s["U"] = torch.empty(S, device="cuda", dtype=torch.float64)
    if case["kind"] == "forces":
        s["nl"].build(s["pos4"], s["L"], T).query(r_list, s["cap"])
        s["pos4"] = pack_positions(_moved(x, s["L"], case["skin"], seed), types)
    return s


# ------------------------------------------------------------------- one pass

def _counts(nl):
    """The rows' lengths, in memory of the caller's own (the library's view ends with its next build)."""
    return nl.neighbors()[1].clone()


def run(s):
    nl, kind = s["nl"], s["kind"]
    if kind == "list":
        if "pos64" in s:
            nl.build_f64(s["pos64"], s["L"], s["T"])
        else:
            nl.build(s["pos4"], s["L"], s["T"])
        nl.query(s["r_list"], s["cap"])
        rows, counts = nl.neighbors()
        return {"counts": counts.clone(), "rows": torch.where(s["column"] < counts[:, None], rows, -1)}
    if kind == "step":
        nl.build(s["pos4"], s["L"], s["T"])
        nl.query_lj_async(s["pos4"], s["r_list"], s["cap"], s["eps"], s["sig"], s["r_cut"], s["e"], s["U"], s["F"])
        return {"counts": _counts(nl), "U": s["U"], "e": s["e"], "F": s["F"]}
    if kind == "train":
        pos4 = pack_positions(s["xyz"], s["types"])
        nl.build_batched(pos4, s["off"], s["Ls"], s["T"])
        nl.query(s["r_list"], s["cap"])
        U = lj_energy(nl, s["xyz"], s["eps"], s["sig"], s["r_cut"], pos4=pos4)
        gx, ge, gs = torch.autograd.grad((U * s["weight"]).sum(), [s["xyz"], s["eps"], s["sig"]])
        return {"counts": _counts(nl), "U": U.detach(), "grad_xyz": gx, "grad_eps": ge, "grad_sig": gs}
    if kind == "ensemble":
        check(s["batch"].run(), "batched step")
    check(qbvh_lj_forward(nl.h, s["pos4"], s["eps"], s["sig"], s["r_cut"], s["e"], s["U"], s["F"], None, None),
          "qbvh_lj_forward")
    out = {"U": s["U"], "e": s["e"], "F": s["F"]}
    if kind == "ensemble":
        out["counts"] = _counts(nl)
    return out


def work(case):
    """Positions read once; the list written once where the pass makes one (read
    once where it is kept), the requested outputs written once.  Arithmetic: 9
    operations per listed pair for its distance, 27 per pair within the cutoff
    for its energy and force."""
    r_list, r_cut, _, _ = _matrices(case)
    n = int(_sizes(case).sum()) if case["kind"] == "ensemble" else case["n"] * case["n_sys"]
    if case["shape"] == "vapor":   # neighbours of the liquid part
        liquid = (case["rho"] - 0.02) / 0.70 * 0.72 / case["rho"]
        listed_, inside = (liquid * _mean_neighbors(case, r[0, 0]) for r in (r_list, r_cut))
    else:
        listed_, inside = (_mean_neighbors(case, r[0, 0]) for r in (r_list, r_cut))
    out = {"list": 0, "step": 16, "forces": 16, "train": 12 + 8, "ensemble": 16}[case["kind"]]
    read = 32 if case["data"] == "f64" else 16
    byts = n * (read + out + 4 + 4 * listed_)
    if case["kind"] == "list":   # the padded matrix a program gets
        byts += n * 4.0 * ((_cap(case, r_list) + 7) // 8 * 8)
    flops = n * (9 * listed_ + (0 if case["kind"] == "list" else 27 * inside))
    return {"bytes": float(byts), "flops": float(flops)}


# ------------------------------------------------------------------- in 64 bits

def _pairs64(x, t, L, rc, eps, sig):
    """Truncated and shifted Lennard-Jones of one system in FP64: per-particle
    energies and forces, and dU/deps, dU/dsigma per type pair, over a cell list
    (all pairs where the box holds fewer than three cells per axis)."""
    n, T = x.shape[0], rc.shape[0]
    e = torch.zeros(n, dtype=torch.float64, device=x.device)
    F = torch.zeros((n, 3), dtype=torch.float64, device=x.device)
    dE = torch.zeros(T * T, dtype=torch.float64, device=x.device)
    dS = torch.zeros(T * T, dtype=torch.float64, device=x.device)
    rc2, ep, sg = ((v.double() if torch.is_tensor(v) else torch.from_numpy(np.asarray(v, np.float64))).to(x.device).reshape(-1)
                   for v in (np.asarray(rc, np.float64) ** 2, eps, sig))
    nc = int(float(L) / float(np.max(rc)))
    if nc < 3:
        nc = 1
    cell3 = torch.clamp((x / L * nc).long(), 0, nc - 1)
    cell = (cell3[:, 0] * nc + cell3[:, 1]) * nc + cell3[:, 2]
    order = cell.argsort()
    count = torch.bincount(cell, minlength=nc ** 3)
    start = count.cumsum(0) - count
    m = int(count.max())
    table = torch.full((nc ** 3, m), -1, dtype=torch.long, device=x.device)
    table[cell[order], torch.arange(n, device=x.device) - start[cell[order]]] = order
    ids = torch.arange(nc ** 3, device=x.device)
    ci = torch.stack([ids // (nc * nc), (ids // nc) % nc, ids % nc], 1)
    chunk = max(1, (1 << 25) // (m * m))
    offsets = [(0, 0, 0)] if nc == 1 else [(a, b, c) for a in (-1, 0, 1) for b in (-1, 0, 1) for c in (-1, 0, 1)]
    rows = table
    sub = max(1, (1 << 25) // m) if nc == 1 else m   # rows of one cell taken at a time
    for o in offsets:
        nb = (ci + torch.tensor(o, device=x.device)) % nc
        nb = (nb[:, 0] * nc + nb[:, 1]) * nc + nb[:, 2]
        for c0 in range(0, nc ** 3, chunk):
            for r0 in range(0, m, sub):
                i, j = rows[c0:c0 + chunk, r0:r0 + sub], table[nb[c0:c0 + chunk]]
                ok = (i[:, :, None] >= 0) & (j[:, None, :] >= 0) & (i[:, :, None] != j[:, None, :])
                ic, jc = i.clamp(min=0), j.clamp(min=0)
                d = [x[jc, k][:, None, :] - x[ic, k][:, :, None] for k in range(3)]
                d = [v - L * torch.round(v / L) for v in d]
                r2 = d[0] * d[0] + d[1] * d[1] + d[2] * d[2]
                if T == 1:
                    p, cut, pe, ps = None, rc2[0], ep[0], sg[0]
                else:
                    p = t[ic][:, :, None] * T + t[jc][:, None, :]
                    cut, pe, ps = rc2[p], ep[p], sg[p]
                ok &= r2 < cut
                r2 = torch.where(ok, r2, cut)
                s, sc = (ps * ps / r2) ** 3, (ps * ps / cut) ** 3
                u = torch.where(ok, 4 * (s * s - s) - 4 * (sc * sc - sc), 0.0)
                w = torch.where(ok, 24 * pe * (2 * s * s - s) / r2, 0.0)
                v = i >= 0
                e.index_add_(0, i[v], 0.5 * (pe * u).sum(2)[v])
                F.index_add_(0, i[v], -torch.stack([(w * d[k]).sum(2) for k in range(3)], -1)[v])
                gs = torch.where(ok, 24 * pe / ps * ((2 * s * s - s) - (2 * sc * sc - sc)), 0.0)
                for q in range(T * T):
                    here = ok if p is None else ok & (p == q)
                    dE[q] += 0.5 * torch.where(here, u, 0.0).sum()
                    dS[q] += 0.5 * torch.where(here, gs, 0.0).sum()
    return e, F, dE.reshape(T, T), dS.reshape(T, T)


def exact(case, seed):
    if case["kind"] == "list":
        return None   # whole numbers only
    _, rc, eps, sig = _matrices(case)
    x, types, off, Ls = _inputs(case, seed)
    if case["kind"] == "forces":
        x = _moved(x, Ls[0], case["skin"], seed)
    got = [_pairs64(x[a:b].double(), types[a:b].long(), L, rc, eps, sig) for a, b, L in zip(off, off[1:], Ls)]
    U = torch.stack([g[0].sum() for g in got])
    if case["kind"] == "train":
        w = torch.linspace(0.5, 1.5, len(Ls), device="cuda", dtype=torch.float64)
        return {"counts": None, "U": U, "grad_xyz": torch.cat([-w[k] * g[1] for k, g in enumerate(got)]),
                "grad_eps": sum(w[k] * g[2] for k, g in enumerate(got)),
                "grad_sig": sum(w[k] * g[3] for k, g in enumerate(got))}
    out = {"U": U, "e": torch.cat([g[0] for g in got]), "F": torch.cat([g[1] for g in got])}
    if case["kind"] != "forces":
        out["counts"] = None
    return out
