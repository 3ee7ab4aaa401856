"""Performance cases of the START radiative-transfer library.

Every case is work a user's program hands to the library through its public
calls (`Context.build_trees`, `set_state`, `rt_solve`, `ionize`, ...):

* ``request``: one served solve, numpy arrays in and out, the trees built for
  it (the serving loop's calls); small ones are bound by latency, launches and
  host round trips, large ones by the march;
* ``batch``: several small requests stacked in one context;
* ``step``: a coupled step of a simulation with static particles and point
  sources, device arrays, the trees kept (optionally with blackbody sources
  and the energy equation, or with resident chains);
* ``h2``: the H2 photodissociation rate over the same chains;
* ``diffuse``: a coupled step with every particle emitting, trees rebuilt and
  the density recomputed as in a run whose particles move;
* ``density``: tree build, neighbour search and SPH density alone.

Inputs are drawn on the GPU from the seed alone: particles on a jittered
lattice (some sites left empty when the count is no cube) with the smoothing
length that holds 32 neighbours, sources uniform in the box, an ionised ball in
a neutral medium.  `exact` restates the method in 64-bit torch: dense over
(virtual source, particle), so only for cases small enough.
"""
import math

import numpy as np
import torch

import paper_1005_5312_gb300 as S

BOX = 6.6                    # kpc
MYR = 3.15576e13             # s
SIGMA, LEN = 6.3e-18, 3.0857e21
ALPHA_A, ALPHA_B = 4.18e-13, 2.59e-13
HNU_L, K_B, T_HI = 13.6 * 1.602176634e-12, 1.380649e-16, 157807.0
KAPPA_LW = 1e-21
DEV = "cuda"


# ------------------------------------------------------------------ the cases
def listed():
    return [
        # a small served request: launches, host round trips and one-block kernels
        dict(name="request-2k", kind="request", n_p=2053, n_s=17, clumpy=False, theta=1.0),
        # an ordinary small request
        dict(name="request-23k", kind="request", n_p=23011, n_s=301, clumpy=True, theta=0.5),
        # the largest served request: 1.7 M particles, tens of thousands of sources
        dict(name="request-1.7m", kind="request", n_p=1700003, n_s=40009, clumpy=False, theta=0.5),
        # sixteen small requests solved with shared launches
        dict(name="batch-16", kind="batch", n_problems=16, n_p=6007, n_s=61, theta=1.0),
        # every source on its own (no cell is accepted): the small plain run
        dict(name="brute-32", kind="step", n_p=32 ** 3, n_s=16, theta=0.0, T_eff=0.0,
             thermal=False, resident=False),
        # the multiple-source run: 64^3 particles, 1024 sources
        dict(name="multisource-64", kind="step", n_p=64 ** 3, n_s=1024, theta=0.5, T_eff=0.0,
             thermal=False, resident=False),
        # blackbody sources with photoheating and the energy equation
        dict(name="thermal-41", kind="step", n_p=41 ** 3, n_s=256, theta=0.5, T_eff=1e5,
             thermal=True, resident=False),
        # later steps of the multiple-source run on resident chains
        dict(name="resident-64", kind="step", n_p=64 ** 3, n_s=1024, theta=0.5, T_eff=0.0,
             thermal=False, resident=True),
        # H2 photodissociation over the same kind of chains, a wide opening angle
        dict(name="h2-50", kind="h2", n_p=50 ** 3, n_s=777, theta=1.0),
        # clump shadowing by recombination photons in their band, a small box
        dict(name="diffuse-clumps-35", kind="diffuse", n_p=35 ** 3, n_s=1, theta=0.7,
             field="clumps", T_rec=1e4, max_pairs=0),
        # the large diffuse run's step at an eighth of its size: log-normal
        # field, 64 sources, split into groups of virtual sources
        dict(name="diffuse-lognormal-128", kind="diffuse", n_p=128 ** 3, n_s=64, theta=0.5,
             field="lognormal", T_rec=0.0, max_pairs=1 << 29),
        # particles that move: trees, neighbour lists and density
        dict(name="density-1m", kind="density", n_p=1048583, n_s=64),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["request", "request", "request", "batch", "step", "step", "step", "h2",
                       "diffuse", "diffuse", "density"])
    theta = rng.choice([0.5, 0.6, 0.7, 0.85, 1.0])
    if kind == "request":
        n_p = _log_int(rng, 2 ** 11, 1_700_000)
        n_s = _log_int(rng, 1, min(n_p, 40_000))
        return dict(kind=kind, n_p=n_p, n_s=n_s, clumpy=rng.random() < 0.5, theta=theta)
    if kind == "batch":
        return dict(kind=kind, n_problems=rng.randint(2, 16), n_p=_log_int(rng, 2 ** 11, 2 ** 14),
                    n_s=_log_int(rng, 1, 500), theta=theta)
    if kind == "step":
        form = rng.choice(["plain", "plain", "brute", "blackbody", "resident"])
        n_p = _log_int(rng, 20 ** 3, 40 ** 3 if form in ("brute", "blackbody") else 64 ** 3)
        n_s = _log_int(rng, 1, 64 if form == "brute" else 300 if form == "blackbody" else 1024)
        return dict(kind=kind, n_p=n_p, n_s=n_s, theta=0.0 if form == "brute" else theta,
                    T_eff=1e5 if form == "blackbody" else 0.0,
                    thermal=form == "blackbody" and rng.random() < 0.5,
                    resident=form == "resident")
    if kind == "h2":
        return dict(kind=kind, n_p=_log_int(rng, 20 ** 3, 64 ** 3), n_s=_log_int(rng, 1, 1024),
                    theta=theta)
    if kind == "diffuse":
        n = int(round(math.exp(rng.uniform(math.log(16), math.log(100)))))
        field = rng.choice(["clumps", "lognormal"])
        return dict(kind=kind, n_p=n ** 3, n_s=1 if field == "clumps" else _log_int(rng, 1, 64),
                    theta=theta, field=field, T_rec=rng.choice([0.0, 1e4]),
                    max_pairs=rng.choice([0, 1 << 29]))
    return dict(kind=kind, n_p=_log_int(rng, 2 ** 13, 2 ** 21), n_s=_log_int(rng, 1, 1024))


# ------------------------------------------------------------------ inputs
def _smoothing(pos, site, n):
    """h with 2h half-way between the 32nd and 33rd neighbour distances.

    The neighbours sit on nearby lattice sites: two sites each way hold them
    unless the particle is near the box's edge or near empty sites, where five
    each way are looked through (then seven)."""
    n_p = pos.shape[1]
    grid = torch.full((n + 14,) * 3, n_p, dtype=torch.int64, device=DEV)
    ijk = torch.stack([site // (n * n), (site // n) % n, site % n]) + 7
    grid[ijk[0], ijk[1], ijk[2]] = torch.arange(n_p, device=DEV)
    flat, stride = grid.reshape(-1), (n + 14) ** 2
    at = ijk[0] * stride + ijk[1] * (n + 14) + ijk[2]
    far = torch.cat([pos, torch.full((3, 1), 1e18, device=DEV)], 1)
    two_h = torch.zeros(n_p, device=DEV)
    dx = BOX / n
    todo = torch.arange(n_p, device=DEV)
    for reach in (2, 5, 7):
        o = torch.arange(-reach, reach + 1, device=DEV)
        off = (o[:, None, None] * stride + o[None, :, None] * (n + 14) + o[None, None, :])
        off = off.reshape(-1)
        off = off[off != 0]
        left = []
        for part in todo.split(max(1, (1 << 25) // off.numel())):
            cand = flat[at[part][:, None] + off[None, :]]
            d2 = sum((far[a][cand] - pos[a][part][:, None]) ** 2 for a in range(3))
            d = torch.topk(d2, 33, dim=1, largest=False, sorted=True).values.sqrt()
            two_h[part] = torch.where(d[:, 32] < 1e8, 0.5 * (d[:, 31] + d[:, 32]),
                                      two_h.new_tensor(4.0 * dx))
            left.append(part[d[:, 32] > (reach + 0.5) * dx])
        todo = torch.cat(left)
        if not todo.numel():
            break
    return 0.5 * two_h


def _particles(n_p, g, adaptive=True):
    """Positions (3, n_p) and h of n_p particles on the smallest jittered
    lattice that holds them, in the lattice's order."""
    n = int(math.ceil(n_p ** (1.0 / 3.0) - 1e-9))
    site = torch.arange(n ** 3, device=DEV)
    if n ** 3 > n_p:
        keep = torch.randperm(n ** 3, generator=g, device=DEV)[:n_p]
        site = torch.sort(keep).values
    dx = BOX / n
    ijk = torch.stack([site // (n * n), (site // n) % n, site % n]).double()
    jit = torch.rand((3, n_p), generator=g, device=DEV, dtype=torch.float64) * 0.5 - 0.25
    pos = ((ijk + 0.5 + jit) * dx).float().contiguous()
    if adaptive:
        h = _smoothing(pos, site, n).float()
    else:
        h = torch.full((n_p,), 1.02 * dx, device=DEV)
    return pos, h, dx


def _ball(pos, inside, outside, r=0.35):
    d2 = sum((pos[a].double() - 0.5 * BOX) ** 2 for a in range(3))
    return torch.where(d2 < (r * BOX) ** 2, d2.new_tensor(inside), d2.new_tensor(outside))


def _clumps(pos, g, bg, dense):
    n_H = torch.full((pos.shape[1],), bg, device=DEV)
    for c in (torch.rand((8, 3), generator=g, device=DEV) * (BOX - 1.6) + 0.8).tolist():
        d2 = sum((pos[a] - c[a]) ** 2 for a in range(3))
        n_H[d2 < 0.64] = dense
    return n_H


def _lognormal(n, g):
    """Mean 1e-3 log-normal density with sigma 1.5 and P(k) ~ k^-3 on n^3 sites."""
    f = torch.fft.rfftn(torch.randn((n, n, n), generator=g, device=DEV, dtype=torch.float64))
    k = torch.fft.fftfreq(n, device=DEV, dtype=torch.float64)
    kz = torch.fft.rfftfreq(n, device=DEV, dtype=torch.float64)
    k2 = k[:, None, None] ** 2 + k[None, :, None] ** 2 + kz[None, None, :] ** 2
    amp = torch.where(k2 > 0, k2.clamp(min=1e-30) ** -0.75, k2.new_tensor(0.0))
    x = torch.fft.irfftn(f * amp, s=(n, n, n)).reshape(-1)
    rho = torch.exp(1.5 * (x - x.mean()) / x.std())
    return (rho * (1e-3 / rho.mean())).float()


def _problem(case, seed, b=0):
    """The inputs of one problem as device tensors."""
    g = torch.Generator(device=DEV)
    g.manual_seed(1_000_003 * (seed % 2_000_003) + 17 * b + 1)
    kind = case["kind"]
    n_p, n_s = case["n_p"], case["n_s"]
    if kind == "batch":   # problems of different sizes
        n_p = max(2, int(n_p * 2.0 ** ((b % 5 - 2) / 2.0)))
        n_s = max(1, int(n_s * (1 + b % 3) / 2))
    pos, h, dx = _particles(n_p, g, adaptive=kind not in ("request", "batch", "density"))
    w = dict(n_p=n_p, n_s=n_s, pos=pos, h=h, V=torch.full((n_p,), dx ** 3, dtype=torch.float64,
                                                          device=DEV))
    w["src_pos"] = (torch.rand((3, n_s), generator=g, device=DEV) * BOX).contiguous()
    w["src_L"] = 1e48 * torch.exp(torch.randn(n_s, generator=g, device=DEV, dtype=torch.float64))
    w["y"] = _ball(pos, 1e-3, 1.0)
    if kind == "diffuse":
        w["src_L"] = torch.full((n_s,), 3e51 if case["field"] == "clumps" else 1e50,
                                dtype=torch.float64, device=DEV)
        if case["field"] == "clumps":
            w["src_pos"] = (torch.full((3, n_s), 0.5 * BOX, device=DEV) +
                            dx * torch.rand((3, n_s), generator=g, device=DEV)).contiguous()
            w["n_H"] = _clumps(pos, g, 2e-4, 0.04)
        else:
            w["n_H"] = _lognormal(int(round(n_p ** (1.0 / 3.0))), g)
        w["y"] = _ball(pos, 1e-3, 1.0 - 1.2e-3)
    elif case.get("clumpy"):
        w["n_H"] = _clumps(pos, g, 2e-4, 0.04)
    else:
        w["n_H"] = torch.full((n_p,), 1e-3, device=DEV)
    w["mass"] = (w["n_H"].double() * w["V"]).float()
    if kind == "density":
        w["mass"] = torch.exp(torch.randn(n_p, generator=g, device=DEV))
    if case.get("thermal"):
        w["T"] = 1e4 * (0.5 + torch.rand(n_p, generator=g, device=DEV, dtype=torch.float64))
    if kind == "h2":
        w["n_H2"] = 1e-4 * torch.exp(1.5 * torch.randn(n_p, generator=g, device=DEV))
    return w


def _params(case):
    p = {}
    if case["kind"] == "step":
        p = dict(T_eff=case["T_eff"], thermal=int(case["thermal"]),
                 reuse_chains=int(case["resident"]))
    elif case["kind"] == "diffuse":
        p = dict(T_rec=case["T_rec"], max_pairs=case["max_pairs"])
    return p


# ------------------------------------------------------------------ the path
def prepare(case, seed):
    kind = case["kind"]
    st = dict(case=case, ctx=S.Context(**_params(case)))
    if kind in ("request", "batch"):
        host = [{k: v.cpu().numpy() if torch.is_tensor(v) else v for k, v in
                 _problem(case, seed, b).items()}
                for b in range(case.get("n_problems", 1))]
        st["problems"] = host
        st["n_H"] = np.concatenate([w["n_H"] for w in host])
        st["y0"] = np.concatenate([w["y"] for w in host])
        return st
    w = _problem(case, seed)
    st.update(w)
    n = w["n_p"]
    st["g"] = torch.zeros(n, dtype=torch.float32, device=DEV)
    st["y1"] = torch.zeros(n, dtype=torch.float64, device=DEV)
    st["rho"] = torch.zeros(n, dtype=torch.float32, device=DEV)
    st["heat"] = torch.zeros(n, dtype=torch.float32, device=DEV)
    st["T1"] = torch.zeros(n, dtype=torch.float64, device=DEV)
    ctx = st["ctx"]
    if kind in ("step", "h2"):   # static particles: the trees are the program's to keep
        ctx.build_trees(w["pos"], w["h"], w["src_pos"], w["src_L"])
    if kind == "step" and case["resident"]:   # the first step finds the chains
        ctx.set_state(w["n_H"], w["y"])
        ctx.rt_solve(case["theta"], gamma_out=st["g"])
    torch.cuda.synchronize()
    return st


def run(st):
    case, ctx = st["case"], st["ctx"]
    kind = case["kind"]
    if kind in ("request", "batch"):
        probs = st["problems"]
        if kind == "batch":
            ctx.build_batch([(w["pos"], w["h"], w["src_pos"], w["src_L"]) for w in probs])
        else:
            w = probs[0]
            ctx.build_trees(w["pos"], w["h"], w["src_pos"], w["src_L"])
        g, y = np.zeros(st["n_H"].shape[0], np.float32), st["y0"].copy()
        ctx.set_state(st["n_H"], y)
        ctx.rt_solve(case["theta"], gamma_out=g)
        ctx.ionize(MYR, y_out=y)
        return [g, y]
    if kind == "h2":
        ctx.h2_dissociation(st["n_H2"], case["theta"], KAPPA_LW, st["g"])
        return st["g"]
    if kind == "density":
        ctx.build_trees(st["pos"], st["h"], st["src_pos"], st["src_L"])
        ctx.sph_density(st["mass"], st["rho"])
        return st["rho"]
    if kind == "diffuse":
        ctx.build_trees(st["pos"], st["h"], st["src_pos"], st["src_L"], st["V"], diffuse=True)
        ctx.sph_density(st["mass"], st["rho"])
        ctx.set_state(st["rho"], st["y"])
        ctx.rt_solve(case["theta"], gamma_out=st["g"])
        out = [st["rho"], st["g"]]
        if case["T_rec"]:
            out.append(ctx.heating(st["heat"]))
        out.append(ctx.ionize(MYR, y_out=st["y1"]))
        return out
    ctx.set_state(st["n_H"], st["y"])
    if case["thermal"]:
        ctx.set_temperature(st["T"])
    ctx.rt_solve(case["theta"], gamma_out=st["g"])
    out = [st["g"]]
    if case["T_eff"]:
        out.append(ctx.heating(st["heat"]))
    out.append(ctx.ionize(MYR, y_out=st["y1"]))
    if case["thermal"]:
        out.append(ctx.temperature(st["T1"]))
    return out


# ------------------------------------------------------------------ work
def _pairs(case):
    """Interaction pairs of a solve (fits to uniform runs)."""
    n_p, n_s, theta = case["n_p"], case["n_s"], case.get("theta", 1.0)
    if theta == 0.0:
        per = n_s
    else:
        per = min(n_s, 14.0 * math.log2(n_s + 1) / theta ** 1.2 + 8.0)
    if case["kind"] == "diffuse":   # and the emitters' cells
        per += min(n_p, 570.0 * (0.5 / theta) ** 1.8 * max(1.0, math.log2(n_p) / 3.0 - 2.9))
    return n_p * case.get("n_problems", 1) * per


def work(case):
    """Inputs read once and results written once; per particle the neighbour
    search's tests, per pair one upstream choice among the few neighbours that
    point towards the source, the link's optical depth and the flux (about 100
    operations)."""
    kind = case["kind"]
    n_p, n_s = case["n_p"] * case.get("n_problems", 1), case["n_s"] * case.get("n_problems", 1)
    build = 16 * n_p + 20 * n_s
    state = 12 * n_p
    out = 12 * n_p
    flops = 100.0 * _pairs(case)
    if kind == "density":
        return dict(bytes=float(build + 8 * n_p), flops=2000.0 * n_p)
    if kind == "h2":
        return dict(bytes=float(8 * n_p), flops=flops)
    if kind == "step" and case["resident"]:
        flops = 40.0 * _pairs(case)   # the links are known
    if kind == "step":
        return dict(bytes=float(state + out), flops=flops)
    if kind == "diffuse":
        build += 20 * n_p             # volumes, masses, density and state
    return dict(bytes=float(build + state + out), flops=flops + 2000.0 * n_p)


def tolerance(case):
    """About four times what the path shows against `exact` (at most 2.4e-7: the
    chain sums are FP32 along tens of links, the decisions those of 64-bit
    arithmetic)."""
    return {"rel": 1e-6}


# ------------------------------------------------------------------ 64-bit reference
def _neighbours(pos, h):
    """(n, K) indices of the particles within 2h, padded with n."""
    n = pos.shape[1]
    p, two_h = pos.double().T.contiguous(), 2.0 * h.double()
    lo = p.min(0).values
    edge = float(two_h.max()) * (1.0 + 1e-9)
    dims = ((p.max(0).values - lo) / edge).long() + 3
    c = ((p - lo) / edge).long() + 1
    cid = (c[:, 0] * dims[1] + c[:, 1]) * dims[2] + c[:, 2]
    order = torch.argsort(cid)
    ncell = int(dims.prod())
    count = torch.bincount(cid, minlength=ncell)
    start = torch.cumsum(count, 0) - count
    m = int(count.max())
    o = torch.arange(-1, 2, device=DEV)
    shift = ((o[:, None, None] * dims[1] + o[None, :, None]) * dims[2] + o[None, None, :]).reshape(-1)
    rows, K = [], 1
    for part in torch.arange(n, device=DEV).split(max(1, (1 << 25) // (27 * m))):
        cell = cid[part][:, None] + shift[None, :]
        slot = torch.arange(m, device=DEV)
        ok = slot[None, None, :] < count[cell][:, :, None]
        k = order[(start[cell][:, :, None] + slot).clamp(max=n - 1)]
        k, ok = k.reshape(len(part), -1), ok.reshape(len(part), -1)
        d2 = sum((p[:, a][k] - p[part, a][:, None]) ** 2 for a in range(3))
        ok &= (d2 < two_h[part][:, None] ** 2) & (k != part[:, None])
        kk = int(ok.sum(1).max())
        K = max(K, kk)
        first = torch.argsort(ok.to(torch.int8), dim=1, descending=True, stable=True)[:, :kk]
        rows.append(torch.where(torch.gather(ok, 1, first), torch.gather(k, 1, first), n))
    nb = torch.full((n, K), n, dtype=torch.int64, device=DEV)
    at = 0
    for r in rows:
        nb[at:at + r.shape[0], :r.shape[1]] = r
        at += r.shape[0]
    return nb


def _density(w, nb):
    p, h = w["pos"].double(), w["h"].double()
    n = w["n_p"]
    m = torch.cat([w["mass"].double(), torch.zeros(1, dtype=torch.float64, device=DEV)])
    rho = torch.zeros(n, dtype=torch.float64, device=DEV)
    far = torch.cat([p, torch.zeros((3, 1), dtype=torch.float64, device=DEV)], 1)
    for part in torch.arange(n, device=DEV).split(1 << 18):
        k = nb[part]
        q = sum((far[a][k] - p[a][part][:, None]) ** 2 for a in range(3)).sqrt() / h[part][:, None]
        wq = torch.where(q < 1, 1 - 1.5 * q ** 2 + 0.75 * q ** 3, 0.25 * (2 - q).clamp(min=0) ** 3)
        rho[part] = (m[part] + (m[k] * wq).sum(1)) / (math.pi * h[part] ** 3)
    return rho


def _octree(pos, L, lo, side):
    """Cells of the octree over one problem's emitters (one member per leaf):
    parent, lower corner, edge, luminosity, float32 centre, member (-1: several)."""
    p = pos.double().T
    q = ((p - lo) * (2097152.0 / side)).floor().clamp(0, 2097151).long()
    key = torch.zeros(p.shape[0], dtype=torch.int64, device=DEV)
    for b in range(21):
        for a in range(3):
            key |= ((q[:, a] >> b) & 1) << (3 * b + 2 - a)
    key, order = torch.sort(key, stable=True)
    members, par_of = order, torch.full_like(order, -1)
    cells = []
    base = 0
    for level in range(22):
        prefix = key >> (3 * (21 - level))
        _, inv, cnt = torch.unique_consecutive(prefix, return_inverse=True, return_counts=True)
        nc = cnt.numel()
        first = torch.cumsum(cnt, 0) - cnt
        Lm, pm = L[members], p[members]
        Ls = torch.zeros(nc, dtype=torch.float64, device=DEV).index_add_(0, inv, Lm)
        M = torch.zeros((nc, 3), dtype=torch.float64, device=DEV).index_add_(0, inv, Lm[:, None] * pm)
        edge = side * 2.0 ** -level
        corner = lo + (q[members[first]] >> (21 - level)).double() * edge
        one = cnt == 1
        cen = torch.where(one[:, None], pm[first], M / Ls[:, None].clamp(min=1e-300))
        cen = torch.where((Ls > 0)[:, None] | one[:, None], cen, corner + 0.5 * edge)
        cells.append(dict(parent=par_of[first], corner=corner,
                          edge=torch.full((nc,), edge, dtype=torch.float64, device=DEV), L=Ls,
                          cen=cen.float().double(), member=torch.where(one, members[first], -1)))
        deeper = ~one[inv]
        if not bool(deeper.any()):
            break
        if level == 21:
            return None
        key, members, par_of = key[deeper], members[deeper], (base + inv)[deeper]
        base += nc
    return {k: torch.cat([c[k] for c in cells]) for k in cells[0]}


def _accepts(t, c, p, theta):
    """(cells c) x (particles): l^2 <= theta^2 d^2, d the distance to the cube."""
    d2 = torch.zeros((c.numel(), p.shape[0]), dtype=torch.float64, device=DEV)
    for a in range(3):
        lw = t["corner"][c, a][:, None]
        d = torch.maximum(lw - p[None, :, a], p[None, :, a] - (lw + t["edge"][c][:, None]))
        d2 += d.clamp(min=0) ** 2
    th = float(np.float32(theta))
    return (t["edge"][c] ** 2)[:, None] <= th * th * d2


def _solve(w, nb, dens, trees, theta, column, reduce):
    """Sum over every target's interaction list.  column: the optical depth (or
    column) per length and density; reduce(tree, r2, tau, L) -> contributions."""
    n = w["n_p"]
    p = w["pos"].double().T.contiguous()
    K = nb.shape[1]
    pad = torch.cat([p, torch.full((1, 3), 1e15, dtype=torch.float64, device=DEV)])
    off = pad[nb] - p[:, None, :]
    unit = off / (off ** 2).sum(2, keepdim=True).sqrt()
    dpad = torch.cat([dens, dens.new_zeros(1)])
    sums = None
    for which, (t, is_self) in enumerate(trees):
        many = torch.arange(t["L"].numel(), device=DEV)
        for c in many.split(max(1, (1 << 27) // (n * K))):
            s = t["cen"][c]
            use = torch.ones((c.numel(), n), dtype=torch.bool, device=DEV)
            par = t["parent"][c]
            has = par >= 0
            if bool(has.any()):
                use[has] = ~_accepts(t, par[has], p, theta)
            several = t["member"][c] < 0
            if bool(several.any()):
                use[several] &= _accepts(t, c[several], p, theta)
            if is_self:
                use &= t["member"][c][:, None] != torch.arange(n, device=DEV)[None, :]
            live = use.any(1)
            if not bool(live.any()):
                continue
            use, s, c = use[live], s[live], c[live]
            b = s[:, None, :] - p[None]
            D = (b ** 2).sum(2)
            Dp = torch.cat([D, D.new_full((D.shape[0], 1), 1e300)], 1)
            closer = Dp[:, nb] < D[:, :, None]
            score = torch.einsum("vnd,nkd->vnk", b, unit)
            score = torch.where(closer, score, score.new_tensor(-1e300))
            best = score.argmax(2)
            end = ~torch.gather(closer, 2, best[:, :, None])[:, :, 0]
            up = torch.gather(nb[None].expand(c.numel(), -1, -1), 2, best[:, :, None])[:, :, 0]
            up = torch.where(end, up.new_tensor(n), up)
            dist = Dp.sqrt()
            dist[:, n] = 0.0
            dl = D.sqrt() - torch.gather(dist, 1, up)
            mean = torch.where(end, dens[None].expand(c.numel(), -1),
                               0.5 * (dens[None] + dpad[up]))
            tau = torch.cat([column * mean * dl, D.new_zeros((c.numel(), 1))], 1)
            nxt = torch.cat([up, up.new_full((c.numel(), 1), n)], 1)
            while bool((nxt[:, :n] < n).any()):
                tau = tau + torch.gather(tau, 1, nxt)
                nxt = torch.gather(nxt, 1, nxt)
            rf = 1e-6 * w["side"]
            out = reduce(which, D.clamp(min=rf * rf), tau[:, :n], t["L"][c][:, None])
            out = [torch.where(use, o, o.new_tensor(0.0)).sum(0) for o in out]
            sums = out if sums is None else [x + y for x, y in zip(sums, out)]
    return sums


def _frame(w):
    p = torch.cat([w["pos"], w["src_pos"]], 1).double()
    lo, hi = p.min(1).values, p.max(1).values
    w["side"] = float((hi - lo).max())
    return lo, w["side"]


def _legendre(lo, hi, n):
    x, wt = np.polynomial.legendre.leggauss(n)
    return 0.5 * (hi + lo) + 0.5 * (hi - lo) * x, 0.5 * (hi - lo) * wt


def _spectrum(T_eff):
    """Nodes u = nu / nu_L and photon weights of a blackbody above the limit."""
    a = HNU_L / (K_B * T_eff)
    u, wt = [], []
    edges = 1.0 + np.concatenate([[0.0], np.geomspace(0.02, 1.0, 12)]) * 80.0 / a
    for lo, hi in zip(edges[:-1], edges[1:]):
        x, q = _legendre(lo, hi, 16)
        u.append(x)
        wt.append(q)
    u, wt = np.concatenate(u), np.concatenate(wt)
    f = wt * u ** 2 / np.expm1(a * u)
    return u, f / f.sum()


def _nodes_sum(tau, u, f):
    """sum f u^-3 e^(-tau u^-3) and the same with (u - 1)."""
    ion, heat = torch.zeros_like(tau), torch.zeros_like(tau)
    for x, q in zip(u.tolist(), f.tolist()):
        v = q * x ** -3 * torch.exp(-tau * x ** -3)
        ion += v
        heat += (x - 1.0) * v
    return ion, heat


def _alpha_B(T):
    l = 2.0 * T_HI / T
    return 2.753e-14 * l ** 1.5 / (1.0 + (l / 2.74) ** 0.407) ** 2.242


def _coll_ion(T):
    l = 2.0 * T_HI / T
    return 21.11 * T ** -1.5 * torch.exp(-0.5 * l) * l ** -1.089 / (1.0 + (l / 0.354) ** 0.874) ** 1.101


def _thermal_step(n_H, y0, T0, k, heat, dt):
    """Case B, point sources: y at the step's first temperature, then the
    implicit energy equation by bisection on ln T."""
    a, c = _alpha_B(T0) * n_H * dt, _coll_ion(T0) * n_H * dt
    b = 1.0 + k * dt + c + 2.0 * a
    y1 = 2.0 * (y0 + a) / (b + (b * b - 4.0 * (a + c) * (y0 + a)).clamp(min=0).sqrt())
    x0, x1 = 1.0 - y0, 1.0 - y1

    def residual(T):
        l = 2.0 * T_HI / T
        rec = 3.435e-30 * T * l ** 1.97 / (1.0 + (l / 2.25) ** 0.376) ** 3.72
        ff = 1.42e-27 * (1.1 + 0.34 * torch.exp(-(5.5 - torch.log10(T)) ** 2 / 3.0)) * T.sqrt()
        exc = 7.5e-19 * torch.exp(-118348.0 / T) / (1.0 + (T / 1e5).sqrt())
        lam = (x1 * n_H) ** 2 * (rec + ff) + x1 * n_H * y1 * n_H * (K_B * T_HI * _coll_ion(T) + exc)
        e = 1.5 * K_B * n_H
        return e * ((1.0 + x1) * T - (1.0 + x0) * T0) + dt * (lam - y1 * n_H * heat)

    lo, hi = torch.full_like(T0, math.log(10.0)), torch.full_like(T0, math.log(1e9))
    for _ in range(100):
        mid = 0.5 * (lo + hi)
        up = residual(torch.exp(mid)) > 0
        lo, hi = torch.where(up, lo, mid), torch.where(up, mid, hi)
    return y1, torch.exp(0.5 * (lo + hi))


def _ionize(n_H, y0, k, alpha, dt):
    A, K = alpha * n_H * dt, k * dt
    disc = (K + 1.0) ** 2 + 4.0 * A * (K + 1.0 - y0)
    return 2.0 * (A + y0) / (2.0 * A + K + 1.0 + disc.sqrt())


def _phi(t):
    return torch.where(t > 0, -torch.expm1(-t) / t.clamp(min=1e-300), t.new_tensor(1.0))


def _point_step(w, theta):
    lo, side = _frame(w)
    nb = _neighbours(w["pos"], w["h"])
    tree = _octree(w["src_pos"], w["src_L"], lo, side)
    n_H = w["n_H"].double()
    dens = (w["y"] * n_H).float().double()
    g, = _solve(w, nb, dens, [(tree, False)], theta, SIGMA * LEN,
                lambda _, r2, tau, L: [L * torch.exp(-tau) / (4 * math.pi * r2 * LEN ** 2)])
    return g, _ionize(n_H, w["y"], SIGMA * g, ALPHA_B, MYR)


def _exact_diffuse(case, w):
    lo, side = _frame(w)
    nb = _neighbours(w["pos"], w["h"])
    rho = _density(w, nb)
    n_H, y0 = rho.float().double(), w["y"]
    dens = (y0 * n_H).float().double()
    ne = (1.0 - y0) * n_H
    a1 = ALPHA_A - ALPHA_B
    L = a1 * ne * ne * w["V"] * LEN ** 3
    trees = [(_octree(w["src_pos"], w["src_L"], lo, side), False),
             (_octree(w["pos"], L, lo, side), True)]
    if trees[1][0] is None:
        return None
    width = K_B * case["T_rec"] / HNU_L
    if width:
        u, q = _legendre(1.0, 1.0 + width, 24)
        q = q / width

    def reduce(which, r2, tau, Lv):
        d = Lv / (4 * math.pi * r2 * LEN ** 2)
        if width and which == 1:
            ion, heat = _nodes_sum(tau, u, q)
            return [d * ion, d * heat]
        return [d * torch.exp(-tau), torch.zeros_like(tau)]

    g, hs = _solve(w, nb, dens, trees, case["theta"], SIGMA * LEN, reduce)
    R = (3.0 * w["V"] / (4.0 * math.pi)) ** (1.0 / 3.0) * LEN
    ts = SIGMA * y0 * n_H * R
    pre = a1 * ne * ne * SIGMA * R
    k = SIGMA * g
    out = [rho, g]
    if width:
        own = [q_ * u_ ** -3 * _phi(ts * u_ ** -3) for u_, q_ in zip(u.tolist(), q.tolist())]
        k = k + pre * sum(own)
        out.append(SIGMA * HNU_L * hs +
                   pre * HNU_L * sum(v * (u_ - 1.0) for v, u_ in zip(own, u.tolist())))
    else:
        k = k + pre * _phi(ts)
    out.append(_ionize(n_H, y0, k, ALPHA_A, MYR))
    return out


def exact(case, seed):
    kind = case["kind"]
    if kind == "diffuse" and case["n_p"] > 36 ** 3:
        return None
    if kind not in ("diffuse", "density"):   # about (virtual sources) x (particles) x 40 candidates
        per = 1.5 * case["n_s"] * case["n_p"] * case.get("n_problems", 1)
        if per > 1.0e8 or (case.get("T_eff") and per > 4e7):
            return None
    with torch.no_grad():
        out = _exact(case, seed)
    if out is None:
        return None
    out = [o.cpu().numpy() for o in out]
    return out[0] if kind in ("h2", "density") else out


def _exact(case, seed):
    kind = case["kind"]
    if kind in ("request", "batch"):
        parts = [_point_step(_problem(case, seed, b), case["theta"])
                 for b in range(case.get("n_problems", 1))]
        return [torch.cat([p[i] for p in parts]) for i in range(2)]
    w = _problem(case, seed)
    if kind == "density":
        return [_density(w, _neighbours(w["pos"], w["h"]))]
    if kind == "diffuse":
        return _exact_diffuse(case, w)
    if kind == "step" and not case["T_eff"]:
        return list(_point_step(w, case["theta"]))
    lo, side = _frame(w)
    nb = _neighbours(w["pos"], w["h"])
    trees = [(_octree(w["src_pos"], w["src_L"], lo, side), False)]
    if kind == "h2":
        def shield(_, r2, N, L):
            x = N / 1e14
            f = torch.where(x <= 1, x.new_tensor(1.0), x.clamp(min=1.0) ** -0.75)
            return [1.13e8 * KAPPA_LW * L / (4 * math.pi * r2 * LEN ** 2) * f]
        return _solve(w, nb, w["n_H2"].double(), trees, case["theta"], LEN, shield)
    u, f = _spectrum(case["T_eff"])
    n_H = w["n_H"].double()

    def band(_, r2, tau, L):
        d = L / (4 * math.pi * r2 * LEN ** 2)
        ion, heat = _nodes_sum(tau, u, f)
        return [d * ion, d * heat]

    g, hs = _solve(w, nb, (w["y"] * n_H).float().double(), trees, case["theta"], SIGMA * LEN, band)
    heat = SIGMA * HNU_L * hs
    if case["thermal"]:
        y1, T1 = _thermal_step(n_H, w["y"], w["T"], SIGMA * g, heat, MYR)
        return [g, heat, y1, T1]
    return [g, heat, _ionize(n_H, w["y"], SIGMA * g, ALPHA_B, MYR)]
