"""Workloads of the halo-finding path, as the programs that use it call it.

A case names one call, or the few that belong together, of the public binding (paper_1110_4372_gb300.rsgpu) on a
catalogue or a set of groups drawn on the GPU from a seed:

    listed()             the fixed cases
    draw(rng)            one more of the same ranges
    prepare(case, seed)  the inputs a program has in hand, and the handles that it keeps
    run(state)           one pass, and what it returns
    work(case)           bytes a pass cannot do without (each input read once, each output written once)
    exact(case, seed)    the computed numbers of a pass in 64 bits, in plain torch

Catalogues follow the recipe of synth.py: NFW halos with dN/dn ~ n^-1.9 from 20 particles up, subhalos, sub-subhalos
in the large boxes, a uniform background, 32^3 particles per (10 Mpc/h)^3, shuffled.  Independent groups follow its
batching-stress recipe: log-uniform sizes, an NFW host with up to 12 co-spatial subhalos moving at 1-3 sigma.
"""
from __future__ import annotations

import ctypes
import math

import numpy as np
import torch

from paper_1110_4372_gb300 import rsgpu

NBAR = 32768 / 10.0 ** 3          # particles per (Mpc/h)^3
HOSTS_PER_PARTICLE = 150_000 / 2 ** 27
DELTA_VIR = 360.0
NN_SUBSET = 10_000                # the paper's subset for groups above 10^4 (Sec. 3.2)
GROUP_BOX = 1000.0


def listed():
    return [
        # 3D groups of one small zoom region or sub-box inside a latency-bound host loop, without allocation
        dict(name="static_4k", kind="static", n=4099, stride=3, b=0.28),
        # the whole path on a small test box: launches and host reads count
        dict(name="find_32k", kind="find", n=32_768, stride=3, b=0.28, f=0.7, min_n=10, subset=0, host=False),
        # the whole path on a 128^3 box
        dict(name="find_2m", kind="find", n=2_097_152, stride=3, b=0.28, f=0.7, min_n=10, subset=0, host=False),
        # the whole path on the 512^3 box, the size the library is quoted on
        dict(name="find_134m", kind="find", n=134_217_728, stride=3, b=0.28, f=0.7, min_n=10, subset=0, host=False),
        # a snapshot in pinned host memory, padded to four floats a row, an odd particle count, labels wanted too
        dict(name="find_host_7m", kind="find", n=7_340_003, stride=4, b=0.28, f=0.7, min_n=10, subset=0, host=True),
        # the paper's subset linking lengths on a 256^3 box
        dict(name="find_subset_17m", kind="find", n=16_777_216, stride=3, b=0.28, f=0.7, min_n=10, subset=NN_SUBSET,
             host=False),
        # a 3D group catalogue alone (labels, then the groups as a list), padded rows
        dict(name="groups3d_33m", kind="groups", n=33_333_333, stride=4, b=0.28, min_n=20),
        # the paper's accelerated 3D FOF on a 128^3 box
        dict(name="accel_2m", kind="accel", n=2_097_152, stride=3, b=0.28, dense_n=16),
        # hierarchies of independent groups of 20 to 50,000 members (a load-balanced worker's share), with the node
        # table and the labels of the first levels
        dict(name="refine_groups", kind="refine", n=9_600_001, nmax=50_000, stride=3, f=0.7, min_n=10, subset=0),
        # the same call on many small groups, where the subtree kernels do the work
        dict(name="refine_small", kind="refine", n=5_000_011, nmax=600, stride=3, f=0.7, min_n=10, subset=0),
        # the halo catalogue of a tree: halo ids, halo table, centres and hosts
        dict(name="catalogue_4m", kind="assign", n=4_194_301, stride=3, f=0.7, min_n=10),
        # unbinding, by the tree above 4096 members (the paper's 4%)
        dict(name="unbind_2m", kind="unbind", n=2_097_152, stride=3, theta=0.04),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["static", "find", "find", "find", "find", "groups", "accel", "refine", "refine", "assign",
                       "unbind"])
    stride = rng.choice([3, 4])
    b = rng.choice([0.2, 0.28, 0.28])
    f = rng.choice([0.5, 0.7, 0.7])
    min_n = rng.choice([10, 10, 20])
    if kind == "static":
        return dict(kind=kind, n=_log_int(rng, 1000, 65_536), stride=stride, b=b)
    if kind == "find":
        return dict(kind=kind, n=_log_int(rng, 4096, 60_000_000), stride=stride, b=b, f=f, min_n=min_n,
                    subset=rng.choice([0, 0, NN_SUBSET]), host=rng.choice([False, False, True]))
    if kind == "groups":
        return dict(kind=kind, n=_log_int(rng, 30_000, 100_000_000), stride=stride, b=b, min_n=min_n)
    if kind == "accel":
        return dict(kind=kind, n=_log_int(rng, 30_000, 8_000_000), stride=stride, b=b, dense_n=rng.choice([8, 16, 32]))
    if kind == "refine":
        n = _log_int(rng, 20_000, 20_000_000)
        return dict(kind=kind, n=n, nmax=_log_int(rng, 200, min(n, 200_000)), stride=stride, f=f, min_n=min_n,
                    subset=rng.choice([0, 0, NN_SUBSET]))
    if kind == "assign":
        return dict(kind=kind, n=_log_int(rng, 30_000, 8_000_000), stride=stride, f=f, min_n=min_n)
    return dict(kind=kind, n=_log_int(rng, 30_000, 2_000_000), stride=stride, theta=rng.choice([0.0, 0.04, 0.04]))


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _sigma1d(mass):
    return 300.0 * (mass / 4000.0) ** (1.0 / 3.0)


def _radius(mass):
    return (3.0 * mass / (4.0 * np.pi * DELTA_VIR * NBAR)) ** (1.0 / 3.0)


def _unit(rng, k):
    d = rng.standard_normal((k, 3))
    return d / np.linalg.norm(d, axis=1, keepdims=True)


def _halo_components(rng, n, box):
    """Hosts, subhalos and sub-subhalos: particle count, mass, centre and bulk velocity of each."""
    nmax = min(1_000_000, max(100, n // 10))
    u = rng.random(max(1, round(HOSTS_PER_PARTICLE * n)))
    a, c = 20.0 ** -0.9, (nmax + 1.0) ** -0.9
    mass = np.floor((a - u * (a - c)) ** (-1.0 / 0.9)).clip(20, nmax)
    mass = mass[np.cumsum(mass) <= 0.8 * n]
    if not len(mass):
        mass = np.array([20.0])
    levels = [dict(n=mass.copy(), mass=mass, centre=rng.random((len(mass), 3)) * box,
                   bulk=rng.standard_normal((len(mass), 3)) * 300.0)]
    for depth in range(0 if n < 1 << 18 else (1 if n < 1 << 23 else 2)):
        up = levels[-1]
        k = rng.integers(1, 9, len(up["mass"])) if depth == 0 else np.where(up["mass"] >= 2000, 2, 0)
        par = np.repeat(np.arange(len(k)), k)
        m = np.floor(rng.uniform(0.01, 0.1, len(par)) * up["mass"][par])
        par, m = par[m >= 10], m[m >= 10]
        at = up["centre"][par] + _unit(rng, len(m)) * (rng.uniform(0.1, 1.0, len(m)) * _radius(up["mass"][par]))[:, None]
        go = up["bulk"][par] + rng.standard_normal((len(m), 3)) * (0.5 * _sigma1d(up["mass"][par]))[:, None]
        up["n"] -= np.bincount(par, weights=m, minlength=len(k))
        levels.append(dict(n=m.copy(), mass=m, centre=at, bulk=go))
    return {q: np.concatenate([lv[q] for lv in levels]) for q in levels[0]}


def _nfw_table(levels=64, grid=2048):
    """Radius over scale radius at enclosed fraction (k / grid)^2, for `levels` concentrations in [5, 15]."""
    c = torch.linspace(5, 15, levels, dtype=torch.float64, device="cuda")[:, None]
    x = torch.cat([torch.zeros(1, dtype=torch.float64, device="cuda"),
                   torch.logspace(-6, 0, 8192, dtype=torch.float64, device="cuda")])[None] * c
    m = torch.log1p(x) - x / (1 + x)
    m = m / m[:, -1:]
    u = (torch.arange(grid + 1, device="cuda", dtype=torch.float64) / grid) ** 2
    u = u[None].expand(levels, -1).contiguous()
    i = torch.searchsorted(m, u).clamp(1, x.shape[1] - 1)
    m0, m1, x0, x1 = m.gather(1, i - 1), m.gather(1, i), x.gather(1, i - 1), x.gather(1, i)
    return c[:, 0], x0 + (x1 - x0) * ((u - m0) / (m1 - m0)).clamp(0, 1)


def _particles(comp, rng, gen, box):
    """Positions (wrapped) and velocities of the components' particles, component by component."""
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a, np.float64)).cuda()  # noqa: E731
    cnt = torch.from_numpy(comp["n"].astype(np.int64)).cuda()
    k = int(comp["n"].sum())
    conc, table = _nfw_table()
    lev = torch.from_numpy(rng.integers(0, len(conc), len(comp["n"]))).cuda()
    scale = dev(_radius(comp["mass"])) / conc[lev]
    sig, centre, bulk = dev(_sigma1d(comp["mass"])).float(), dev(comp["centre"]), dev(comp["bulk"]).float()
    pos = torch.empty((k, 3), dtype=torch.float32, device="cuda")
    vel = torch.empty((k, 3), dtype=torch.float32, device="cuda")
    owner = torch.repeat_interleave(torch.arange(len(cnt), device="cuda"), cnt)
    for a in range(0, k, 1 << 24):
        o = owner[a:a + (1 << 24)]
        s = torch.rand(len(o), generator=gen, device="cuda", dtype=torch.float64).sqrt() * (table.shape[1] - 1)
        i = s.long().clamp(max=table.shape[1] - 2)
        lo = table[lev[o], i]
        r = (lo + (table[lev[o], i + 1] - lo) * (s - i)) * scale[o]
        d = torch.randn((len(o), 3), generator=gen, device="cuda")
        d /= d.norm(dim=1, keepdim=True).clamp(min=1e-12)
        x = torch.remainder(centre[o] + d.double() * r[:, None], box).float()
        pos[a:a + len(o)] = torch.where(x >= box, torch.zeros_like(x), x)
        vel[a:a + len(o)] = bulk[o] + torch.randn((len(o), 3), generator=gen, device="cuda") * sig[o][:, None]
    return pos, vel, owner


def _rows(a, stride):
    return a.contiguous() if stride == 3 else torch.nn.functional.pad(a, (0, 1)).contiguous()


def _catalogue(n, stride, seed):
    box = float(np.float32(10.0 * (n / 32768) ** (1.0 / 3.0)))
    rng = np.random.default_rng([seed, n])
    gen = torch.Generator(device="cuda").manual_seed(int(rng.integers(1 << 62)))
    hp, hv, _ = _particles(_halo_components(rng, n, box), rng, gen, box)
    k = n - len(hp)
    bg = torch.rand((k, 3), generator=gen, device="cuda") * box
    bg = torch.where(bg >= box, torch.zeros_like(bg), bg)
    bv = torch.randn((k, 3), generator=gen, device="cuda") * 20.0
    mix = torch.randperm(n, generator=gen, device="cuda")
    return _rows(torch.cat([hp, bg])[mix], stride), _rows(torch.cat([hv, bv])[mix], stride), box


def _independent_groups(n, nmax, stride, seed):
    rng = np.random.default_rng([seed, n, nmax])
    gen = torch.Generator(device="cuda").manual_seed(int(rng.integers(1 << 62)))
    mean = (nmax - 20) / math.log(nmax / 20)
    size = np.exp(rng.uniform(math.log(20), math.log(nmax + 1), int(4 * n / mean) + 64)).astype(np.int64).clip(20, nmax)
    size = size[:1 + int(np.searchsorted(np.cumsum(size), n - 20))]
    size[-1] += n - size.sum()                              # n members in all
    groups = len(size)
    sub = np.floor(rng.uniform(0.01, 0.1, (groups, 12)) * size[:, None])
    sub[(np.arange(12)[None] >= rng.integers(0, 13, groups)[:, None]) | (sub < 10)] = 0
    host = size - sub.sum(1)
    part = np.concatenate([host[:, None], sub], 1)          # (groups, 13)
    mass = np.concatenate([size[:, None], sub], 1)
    bulk = np.repeat(rng.standard_normal((groups, 1, 3)) * 300.0, 13, 1)
    speed = rng.uniform(1, 3, (groups, 12)) * _sigma1d(size)[:, None]
    bulk[:, 1:] += _unit(rng, groups * 12).reshape(groups, 12, 3) * speed[..., None]
    centre = np.repeat(rng.random((groups, 1, 3)) * GROUP_BOX, 13, 1)
    keep = part.reshape(-1) > 0
    comp = dict(n=part.reshape(-1)[keep], mass=mass.reshape(-1)[keep], centre=centre.reshape(-1, 3)[keep],
                bulk=bulk.reshape(-1, 3)[keep])
    pos, vel, owner = _particles(comp, rng, gen, GROUP_BOX)
    group = torch.from_numpy(np.repeat(np.arange(groups), 13)[keep]).cuda()[owner]
    mix = (group + torch.rand(len(pos), generator=gen, device="cuda", dtype=torch.float64)).argsort()
    off = torch.from_numpy(np.concatenate([[0], np.cumsum(size)])).cuda()
    return _rows(pos[mix], stride), _rows(vel[mix], stride), off


_kept = {}


def _context():
    """The one context a program keeps for all its catalogues."""
    if "ctx" not in _kept:
        _kept["ctx"] = rsgpu.Context()
    return _kept["ctx"]


def _static_call():
    fn = rsgpu.lib().rs_fof3d_static
    fn.restype = ctypes.c_int
    fn.argtypes = [ctypes.c_void_p, ctypes.c_int32, ctypes.c_int64, ctypes.c_double, ctypes.c_double, ctypes.c_void_p,
                   ctypes.c_void_p]
    return fn


def prepare(case, seed):
    s = dict(case, ctx=_context(), kept={})
    if case["kind"] == "refine":
        s["pos"], s["vel"], s["offsets"] = _independent_groups(case["n"], case["nmax"], case["stride"], seed)
        s["box"] = GROUP_BOX
        s["perm"] = torch.arange(len(s["pos"]), dtype=torch.int32, device="cuda")
        return s
    n = case["n"]
    s["pos"], s["vel"], s["box"] = _catalogue(n, case["stride"], seed)
    if case["kind"] in ("static", "groups", "accel", "find"):
        s["labels"] = torch.empty(n, dtype=torch.int32, device="cuda")
    if case["kind"] == "static":
        s["call"] = _static_call()
    if case["kind"] == "find":
        s["halo_id"] = torch.empty(n, dtype=torch.int32, device="cuda")
        s["params"] = rsgpu.params(b=case["b"], f=case["f"], min_n=case["min_n"], nn_subset=case["subset"],
                                   nn_seed=11104372)
        if case["host"]:
            for k in ("pos", "vel", "labels", "halo_id"):
                s[k] = s[k].cpu().pin_memory()
    if case["kind"] in ("assign", "unbind"):
        f, min_n = case.get("f", 0.7), case.get("min_n", 10)
        s["params"] = p = rsgpu.params(f=f, min_n=min_n)
        ctx = s["ctx"]
        labels, _, _ = rsgpu.rs_fof3d(ctx, s["pos"], s["box"], p.b)
        perm, off = rsgpu.rs_group_sort(ctx, labels, min_n)
        s["tree"] = rsgpu.rs_refine6d(ctx, s["pos"], s["vel"], s["box"], perm, off, f, min_n)
        s["nodes"] = s["tree"].nodes()
    if case["kind"] == "unbind":
        s["hid"], s["halos"] = rsgpu.rs_assign_ex(ctx, s["tree"], s["pos"], s["vel"], s["box"], p)
        s["host"] = rsgpu.rs_halo_props(ctx, s["tree"], s["halos"], s["hid"])["host"]
        s["gm"] = rsgpu.particle_gm(NBAR)
    return s


# ---------------------------------------------------------------------------
# passes
# ---------------------------------------------------------------------------
# what a whole-path call reports about its catalogue (the other fields say how the work was split)
FOUND = ("n_fof_groups", "n_members", "n_nodes", "n_levels", "n_seeds", "n_halos", "n_tieband6d", "sum_level_members")


LEVELS = 8  # levels whose labels a refinement's user asks for


def _keep(s, **found):
    """Results of a length that the data decide, in buffers of the program's own (zeros after the last row): no
    particle list is longer than n, and n / 10 rows hold every table of nodes, groups or halos here."""
    out = {}
    for k, v in found.items():
        if k not in s["kept"]:
            rows = s["n"] if k in PER_PARTICLE else s["n"] // 10 + 64
            s["kept"][k] = torch.zeros((rows,) + v.shape[1:], dtype=v.dtype, device=v.device)
        out[k] = s["kept"][k]
        out[k][:len(v)] = v
    return out


PER_PARTICLE = ("perm", "halo_id", "bound_own", "phi_own")


def _node_table(tree):
    """The node table in (level, smallest member) order, the order a catalogue is written in."""
    nd = tree.nodes()
    order = ((nd["level"].long() << 32) | nd["minidx"].long()).argsort()
    at = torch.empty_like(order)
    at[order] = torch.arange(len(order), device=order.device)
    out = {k: v[order] for k, v in nd.items()}
    out["parent"] = torch.where(out["parent"] >= 0, at[out["parent"].long().clamp(min=0)], -1)
    return out


def run(s):
    kind, ctx = s["kind"], s["ctx"]
    if kind == "static":
        st = s["call"](s["pos"].data_ptr(), s["stride"], s["n"], s["box"], s["b"], s["labels"].data_ptr(),
                       torch.cuda.current_stream().cuda_stream)
        return [s["labels"], int(st)]
    if kind == "find":
        hid, labels, stats = rsgpu.rs_find_halos(ctx, s["pos"], s["vel"], s["box"], s["params"], s["labels"],
                                                 s["halo_id"])
        return [hid, labels, {k: stats[k] for k in FOUND}]
    if kind == "groups":
        labels, n_groups, _ = rsgpu.rs_fof3d(ctx, s["pos"], s["box"], s["b"], s["labels"], want_groups=True)
        perm, off = rsgpu.rs_group_sort(ctx, labels, s["min_n"])
        return [labels, n_groups, _keep(s, perm=perm, offsets=off), len(off) - 1, len(perm)]
    if kind == "accel":
        return list(rsgpu.rs_fof3d_accel(ctx, s["pos"], s["box"], s["b"], s["dense_n"], s["labels"]))
    if kind == "refine":
        tree = rsgpu.rs_refine6d_sampled(ctx, s["pos"], s["vel"], s["box"], s["perm"], s["offsets"], s["f"],
                                         s["min_n"], s["subset"], 11104372)
        info = tree.info()
        return [_keep(s, **_node_table(tree)), [tree.level_labels(k) for k in range(LEVELS)], info.n_nodes,
                info.n_levels, info.n_seeds, info.n_tieband]
    if kind == "assign":
        hid, halos = rsgpu.rs_assign_ex(ctx, s["tree"], s["pos"], s["vel"], s["box"], s["params"])
        hp = rsgpu.rs_halo_props(ctx, s["tree"], halos, hid)
        c = hp.pop("centre_node").long()  # a node's own name is its level and smallest member
        return _keep(s, **halos.arrays(), **hp, halo_id=hid, centre_level=s["nodes"]["level"][c],
                     centre_minidx=s["nodes"]["minidx"][c])
    return _keep(s, **rsgpu.rs_unbind(ctx, s["tree"], s["halos"], s["hid"], s["host"], s["pos"], s["vel"], s["gm"],
                                      0.0, s["theta"]))


def work(case):
    # a row's positions (and velocities), the indices or ids that go in, and what comes out per particle
    per = {"static": 12 + 4, "groups": 12 + 4 + 4, "accel": 12 + 4, "find": 24 + 4 + 4, "assign": 24 + 4 + 4,
           "unbind": 24 + 4 + 1 + 8, "refine": 24 + 4 + 4 * LEVELS}[case["kind"]]
    return dict(bytes=case["n"] * per, flops=0)


# ---------------------------------------------------------------------------
# computed numbers in 64 bits (labels, ids and counts have none)
# ---------------------------------------------------------------------------
def exact(case, seed):
    if case["kind"] == "assign":
        s = prepare(case, seed)
        return _keep(s, **_exact_table(s))
    if case["kind"] == "unbind":
        s = prepare(case, seed)
        return _keep(s, **_exact_unbind(s))
    # labels, ids and counts; or a whole hierarchy, which plain torch takes minutes for
    return None


def _image(d, box):
    return d - box * torch.round(d / box)


def _exact_table(s):
    """The halo table of a tree (Sec. 3.3): seeds merged by Eq. 2, means and dispersions of the merged seeds'
    members, r_dyn,vir^2 by Eq. 4."""
    nd, box, n = s["nodes"], s["box"], s["n"]
    mem = s["tree"].members().long()
    pos, vel = s["pos"][:, :3].double(), s["vel"][:, :3].double()
    root = torch.arange(len(nd["parent"]), device="cuda")
    for _ in range(int(nd["level"].max())):
        root = torch.where(nd["parent"][root] >= 0, nd["parent"][root].long(), root)
    leaf = (nd["nchild"] == 0).nonzero()[:, 0]
    leaf = leaf[nd["first"][leaf].argsort()]
    root = root[leaf]
    g = {k: nd[k][leaf] for k in ("count", "minidx", "first", "xbar", "vbar", "sigx", "sigv")}
    L = len(leaf)
    ratio = lambda a, b: torch.where(b > 0, a / b, torch.where(a > 0, math.inf, 0.0))  # noqa: E731
    edges = []
    for d in range(1, L):
        a = (root[:-d] == root[d:]).nonzero()[:, 0]
        if not len(a):
            break
        b = a + d
        a_small = torch.where(g["count"][a] != g["count"][b], g["count"][a] < g["count"][b],
                              g["minidx"][a] > g["minidx"][b])
        q = torch.where(a_small, a, b)
        mu = lambda t: t[q] ** 2 / g["count"][q]  # noqa: E731
        dx2 = (_image(g["xbar"][a] - g["xbar"][b], box) ** 2).sum(1)
        dv2 = ((g["vbar"][a] - g["vbar"][b]) ** 2).sum(1)
        e = (ratio(dx2, mu(g["sigx"])) + ratio(dv2, mu(g["sigv"]))).sqrt() < s["params"].merge_thresh
        edges.append(torch.stack([a[e], b[e]]))
    lab = torch.arange(L, device="cuda")
    if edges:
        a, b = torch.cat(edges, 1)
        while True:
            low = torch.minimum(lab[a], lab[b])
            new = lab.clone().scatter_reduce_(0, a, low, "amin").scatter_reduce_(0, b, low, "amin")
            new = new[new]
            if torch.equal(new, lab):
                break
            lab = new
    head, halo = lab.unique(return_inverse=True)
    H = len(head)
    cnt = g["count"]
    owner = torch.repeat_interleave(torch.arange(L, device="cuda"), cnt)
    within = torch.arange(len(owner), device="cuda") - (cnt.cumsum(0) - cnt)[owner]
    p = mem[g["first"][owner] + within]
    h = halo[owner]
    num = torch.bincount(h, minlength=H).double()
    mean = lambda t: torch.zeros((H, 3), dtype=torch.float64, device="cuda").index_add_(0, h, t) / num[:, None]  # noqa: E731
    ref = pos[mem[g["first"][head]]]
    xbar = torch.remainder(ref + mean(_image(pos[p] - ref[h], box)), box)
    v0 = vel[mem[g["first"][head]]]
    vbar = v0 + mean(vel[p] - v0[h])
    sigv = mean((vel[p] - vbar[h]) ** 2).sum(1).sqrt()
    r = _image(pos[p] - xbar[h], box).norm(dim=1)
    o = r.argsort(stable=True)
    o = o[h[o].argsort(stable=True)]
    start = (num.cumsum(0) - num)[h[o]]
    k = torch.arange(1, len(o) + 1, device="cuda") - start
    best = torch.zeros(H, dtype=torch.float64, device="cuda")
    best.scatter_reduce_(0, h[o], torch.where(r[o] > 0, k / r[o], 0.0), "amax")
    rho = 4.0 / 3.0 * math.pi * s["params"].delta_vir * n / box ** 3
    return dict(xbar=xbar, vbar=vbar, sigv=sigv, rdyn2=best / rho)


def _exact_unbind(s):
    """Bulk velocity of every halo's set and every particle's potential in its own halo's set (App. B, summed
    directly)."""
    hid, host, box, n = s["hid"].long(), s["host"].long(), s["box"], s["n"]
    ids = s["halos"].arrays()["id"].long()
    H = len(ids)
    sid, order = ids.sort()
    rank = lambda i: torch.where(i >= 0, order[torch.searchsorted(sid, i.clamp(min=0)).clamp(max=H - 1)], -1)  # noqa: E731
    up = rank(host)
    part = (hid >= 0).nonzero()[:, 0]
    at, rows = rank(hid[part]), []
    while len(part):
        rows.append(torch.stack([at, part]))
        at = up[at]
        part, at = part[at >= 0], at[at >= 0]
    r, p = torch.cat(rows, 1)
    o = r.argsort(stable=True)
    r, p = r[o], p[o]
    num = torch.bincount(r, minlength=H)
    pos, vel = s["pos"][:, :3].double(), s["vel"][:, :3].double()
    vbulk = torch.zeros((H, 3), dtype=torch.float64, device="cuda").index_add_(0, r, vel[p])
    vbulk /= num.clamp(min=1)[:, None]
    phi = torch.full((n,), math.nan, dtype=torch.float64, device="cuda")
    ends = num.cumsum(0).tolist()
    for k, (size, end, halo) in enumerate(zip(num.tolist(), ends, ids.tolist())):
        q = p[end - size:end]
        x = _image(pos[q] - pos[q[:1]], box)
        own = (hid[q] == halo).nonzero()[:, 0]
        step = max(1, (1 << 25) // max(size, 1))
        for a in range(0, len(own), step):
            t = own[a:a + step]
            d2 = ((x[t, 0, None] - x[None, :, 0]) ** 2 + (x[t, 1, None] - x[None, :, 1]) ** 2
                  + (x[t, 2, None] - x[None, :, 2]) ** 2)
            w = d2.rsqrt_()
            w[torch.isinf(w)] = 0.0
            phi[q[t]] = -s["gm"] * w.sum(1)
    return dict(phi_own=phi, vbulk=vbulk)
