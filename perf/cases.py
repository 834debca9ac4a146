"""Performance cases of the SPH neighbour loops: the calls a simulation code makes, over the
sizes, gas distributions and options it makes them with, and what they return in 64 bits.

A case is a dict of plain values:
  kind    "step"    one kick-drift-kick step of one simulation (sph_step), the state moving on
          "sphenix" the same with the SPHENIX flavour (sph_step_sphenix)
          "loops"   sph_build_cells, sph_density and sph_force on given particles
          "masked"  the same with the loops on an active subset (a sub-step's work)
          "pool"    one sph_step of many boxes together
          "fof"     friends-of-friends groups
  gas     "lattice" jittered lattice, "clustered" Plummer spheres plus a uniform background,
          "spheres" two uniform spheres in a large empty box, "boxes" uneven boxes of a pool
  n       particles (a cube for a lattice), or boxes for a pool, whose sizes run from n_min to
          n_max, log-uniform
  nested  nested grids instead of the uniform grid; margin, n_leaf, kernel: sph_params
"""
import math

import torch

from paper_2305_13380_gb300 import sph

ETA = 1.2348
GAMMA_K = (1.825742, 2.018932, 1.936492)  # support over h: cubic, quartic, Wendland C2
BETA_V, ALPHA_V, EPS_B, GAMMA, CFL = 3.0, 0.8, 1e-4, 5.0 / 3.0, 0.1
POS = ("x", "y", "z")
STATE = POS + ("vx", "vy", "vz", "u", "h") + sph.FORCE_FIELDS + ("rho", "f", "div_v", "curl_v", "P", "c", "balsara")


def _case(kind, gas, n, nested=False, kernel=0, **more):
    # the margin and leaf size that the autotuner settles on for large inputs, unless given
    return {"kind": kind, "gas": gas, "n": n, "nested": nested, "kernel": kernel,
            "margin": 0.03 if nested or n > 1000000 else 0.05, "n_leaf": 32 if nested else 16, **more}


def listed():
    return [
        # the smallest plain step: one 16^3 box, where launches and latency are what counts
        {"name": "step_lattice_4096", **_case("step", "lattice", 16 ** 3)},
        # a small served request: two spheres of a few thousand particles in a large box
        {"name": "loops_spheres_6k", **_case("loops", "spheres", 6007, nested=True)},
        # the first evaluation of a mid-sized box, odd side, from the lattice's guess of h
        {"name": "loops_lattice_227k", **_case("loops", "lattice", 61 ** 3)},
        # the headline step: 128^3 particles of nearly uniform gas
        {"name": "step_lattice_2m", **_case("step", "lattice", 128 ** 3)},
        # the clustered box: 64 Plummer spheres, smoothing lengths over two decades
        {"name": "loops_clustered_2m", **_case("loops", "clustered", 2 ** 21, nested=True)},
        # a large served request, an odd count
        {"name": "loops_spheres_400k", **_case("loops", "spheres", 400003, nested=True)},
        # a batch of uneven boxes, lattice and clustered in turn, accelerations taken anew
        {"name": "pool_boxes_48", **_case("pool", "boxes", 48, nested=True, n_min=1000, n_max=30000)},
        # a batch of lattice boxes stepped together from a captured CUDA graph
        {"name": "pool_lattices_64", **_case("pool", "lattices", 64, n_min=1000, n_max=30000)},
        # the production flavour: viscosity switch and conduction, a third neighbour loop
        {"name": "sphenix_lattice_885k", **_case("sphenix", "lattice", 96 ** 3)},
        # a wider kernel on clustered gas
        {"name": "loops_wendland_300k", **_case("loops", "clustered", 300007, nested=True, kernel=2)},
        # a sub-step of the time-step hierarchy: the densest tenth of a clustered box
        {"name": "masked_clustered_1m", **_case("masked", "clustered", 1000003, nested=True, share=0.1)},
        # group finding at the usual fifth of the mean spacing
        {"name": "fof_clustered_1m", **_case("fof", "clustered", 2 ** 20)},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    what = rng.choice(["step", "step", "loops", "loops", "loops", "loops", "spheres", "pool", "sphenix", "masked", "fof"])
    if what in ("step", "sphenix"):
        return _case(what, "lattice", _log(rng, 10, 128 if what == "step" else 96) ** 3)
    if what == "loops":
        kernel = rng.choice([0, 0, 0, 1, 2])
        if rng.random() < 0.4:
            return _case("loops", "lattice", _log(rng, 9, 110) ** 3, kernel=kernel)
        return _case("loops", "clustered", _log(rng, 4000, 2 ** 21 if kernel == 0 else 400000), nested=True, kernel=kernel)
    if what == "spheres":
        return _case("loops", "spheres", _log(rng, 1000, 500000), nested=True)
    if what == "pool":
        nested = rng.random() < 0.5
        return _case("pool", "boxes" if nested else "lattices", _log(rng, 4, 64), nested=nested, n_min=1000,
                     n_max=_log(rng, 4000, 30000))
    if what == "masked":
        share = math.exp(rng.uniform(math.log(0.01), math.log(0.5)))
        if rng.random() < 0.5:
            return _case("masked", "lattice", _log(rng, 20, 128) ** 3, share=share)
        return _case("masked", "clustered", _log(rng, 20000, 1000000), nested=True, share=share)
    return _case("fof", "clustered", _log(rng, 10000, 2 ** 21))


# ---- inputs ------------------------------------------------------------------

def _gen(seed, k=0):
    return torch.Generator(device="cuda").manual_seed((seed * 1000003 + k * 7919 + 12345) % (1 << 62))


def _uni(g, n):
    return torch.rand(n, generator=g, dtype=torch.float64, device="cuda")


def _nor(g, n):
    return torch.randn(n, generator=g, dtype=torch.float64, device="cuda")


def _directions(g, n):
    cth, phi = 2 * _uni(g, n) - 1, 2 * math.pi * _uni(g, n)
    sth = torch.sqrt(torch.clamp(1 - cth * cth, min=0.0))
    return torch.stack([sth * torch.cos(phi), sth * torch.sin(phi), cth])


def _fields(pos, L, vel, u, h0):
    """Positions wrapped into [0, L) in 64 bits, the other fields in 32, equal masses summing to 1."""
    n = pos.shape[1]
    pos = torch.remainder(pos, L)
    pos = torch.where(pos >= L, pos - L, pos)
    p = {k: pos[i].contiguous() for i, k in enumerate(POS)}
    p.update({k: vel[i].float().contiguous() for i, k in enumerate(("vx", "vy", "vz"))})
    p["m"] = torch.full((n,), 1.0 / n, dtype=torch.float32, device="cuda")
    p["u"] = u.float().contiguous()
    p["h0"] = h0.float().contiguous()
    return p


def _lattice(n, g):
    """Jittered lattice in the unit box: +-0.1 spacings, u = 1 +- 1 %, velocities N(0, 0.01^2)."""
    side = round(n ** (1 / 3))
    d = 1.0 / side
    i = torch.arange(n, device="cuda")
    ijk = torch.stack([i % side, (i // side) % side, i // (side * side)]).double()
    pos = (ijk + 0.5 + 0.1 * (2 * _uni(g, 3 * n).view(3, n) - 1)) * d
    u = 1 + 0.01 * (2 * _uni(g, n) - 1)
    return _fields(pos, 1.0, 0.01 * _nor(g, 3 * n).view(3, n), u, torch.full((n,), ETA * d, device="cuda"))


def _clustered(n, g, spheres=None, frac=0.7):
    """70 % in Plummer spheres (scale radii log-uniform in 0.002-0.02), 30 % uniform, unit box;
    u log-normal, velocities N(0, 0.05^2); h0 from the spheres' own density."""
    spheres = spheres or (4 if n < 100000 else 64)
    ncl = int(round(frac * n))
    own = torch.arange(ncl, device="cuda") * spheres // max(ncl, 1)
    per = torch.bincount(own, minlength=spheres).double()
    a = 0.002 * 10 ** _uni(g, spheres)
    cen = _uni(g, 3 * spheres).view(3, spheres)
    X = _uni(g, ncl).clamp(1e-12, 1 - 1e-9)
    r = a[own] / torch.sqrt(X ** (-2 / 3) - 1)
    pos = torch.cat([cen[:, own] + r * _directions(g, ncl), _uni(g, 3 * (n - ncl)).view(3, n - ncl)], 1)
    dens = torch.full((n,), float(n - ncl), dtype=torch.float64, device="cuda")
    dens[:ncl] += 3 * per[own] / (4 * math.pi * a[own] ** 3) * (1 + (r / a[own]) ** 2) ** -2.5
    h0 = torch.clamp(ETA * dens ** (-1 / 3), max=0.1)
    return _fields(pos, 1.0, 0.05 * _nor(g, 3 * n).view(3, n), torch.exp(_nor(g, n)), h0)


def _spheres(n, g):
    """Two uniform spheres (radii 0.1-0.3) approaching along x in a box of side 2, u = 0.05."""
    rr = [float(v) for v in _uni(g, 3)]
    r1, r2, vrel = 0.1 + 0.2 * rr[0], 0.1 + 0.2 * rr[1], 0.5 + 1.5 * rr[2]
    n1 = min(n - 1, max(1, round(n * r1 ** 3 / (r1 ** 3 + r2 ** 3))))
    first = torch.arange(n, device="cuda") < n1
    half = 0.5 * (r1 + r2 + 0.05)
    rad = torch.where(first, r1, r2) * _uni(g, n) ** (1 / 3)
    pos = rad * _directions(g, n) + 1.0
    pos[0] += torch.where(first, -half, half)
    vel = torch.zeros(3, n, dtype=torch.float64, device="cuda")
    vel[0] = torch.where(first, 0.5 * vrel, -0.5 * vrel)
    dens = n / (4 / 3 * math.pi * (r1 ** 3 + r2 ** 3))
    return _fields(pos, 2.0, vel, torch.full((n,), 0.05, device="cuda"),
                   torch.full((n,), ETA * dens ** (-1 / 3), device="cuda"))


def _box_sizes(case):
    """Counts of a pool's boxes: log-uniform from n_min to n_max, every box another; cubes for lattices."""
    out = []
    for b in range(case["n"]):
        s = case["n_min"] * (case["n_max"] / case["n_min"]) ** (((b * 0.6180339887498949) + 0.5) % 1.0)
        lattice = case["gas"] == "lattices" or b % 2 == 0
        out.append((lattice, max(4, round(s ** (1 / 3))) ** 3 if lattice else int(s)))
    return out


def _inputs(case, seed):
    """(particles, box side, box of each particle or None, offsets of the boxes)."""
    n, gas = case["n"], case["gas"]
    if gas in ("boxes", "lattices"):
        boxes, sizes = [], _box_sizes(case)
        for b, (lattice, nb) in enumerate(sizes):
            g = _gen(seed, b + 1)
            # a box keeps at least 800 background particles, so that no support nears half its side
            boxes.append(_lattice(nb, g) if lattice else _clustered(nb, g, 4, min(0.7, 1 - 800 / nb)))
        p = {k: torch.cat([q[k] for q in boxes]) for k in boxes[0]}
        counts = torch.tensor([nb for _, nb in sizes])
        sim = torch.repeat_interleave(torch.arange(len(sizes)), counts).cuda()
        return p, 1.0, sim, torch.cat([torch.zeros(1, dtype=torch.int64), counts.cumsum(0)]).cuda()
    p = {"lattice": _lattice, "clustered": _clustered, "spheres": _spheres}[gas](n, _gen(seed))
    return p, 2.0 if gas == "spheres" else 1.0, None, torch.tensor([0, n], device="cuda")


def _active(case, p):
    """The particles a sub-step updates: the smallest supports, or a ball about the centre of a lattice."""
    n = p["x"].shape[0]
    rank = p["h0"].double()
    if case["gas"] == "lattice":
        rank = sum((p[k] - 0.5) ** 2 for k in POS)
    on = torch.zeros(n, dtype=torch.uint8, device="cuda")
    on[torch.argsort(rank)[:max(1, int(case["share"] * n))]] = 1
    return on


def _sphenix_start(seed, n):
    g = _gen(seed, 999)
    return (0.1 + 0.4 * _uni(g, n)).float(), (0.2 * _uni(g, n)).float()


def _params(case, L, flags=0):
    return sph.sph_default_params(box_size=L, cell_margin=case["margin"], n_leaf=case["n_leaf"], kernel=case["kernel"],
                                  flags=flags | (sph.SPH_FLAG_TREE if case["nested"] else 0))


# ---- a pass ------------------------------------------------------------------

def prepare(case, seed):
    p, L, _, off = _inputs(case, seed)
    n, kind = p["x"].shape[0], case["kind"]
    s = {"case": case}
    if kind in ("step", "sphenix", "pool"):
        # the pool's arrays, started as a user's program starts them: one synchronous step with dt = 0
        a = {k: p[k] for k in POS + ("vx", "vy", "vz", "u", "m")}
        a.update({k: torch.zeros(n, dtype=torch.float32, device="cuda") for k in STATE if k not in a})
        a["h"] = p["h0"].clone()
        sims = off.shape[0] - 1
        a["dt"] = torch.zeros(sims, dtype=torch.float64, device="cuda")
        s["pool"] = sph.pool(off, torch.full((sims,), L, dtype=torch.float64, device="cuda"), a)
        s["out"] = {k: a[k] for k in STATE}
        stream = torch.cuda.Stream() if case["gas"] == "lattices" else torch.cuda.current_stream()
        stream.wait_stream(torch.cuda.current_stream())
        first = sph.Context(_params(case, L, sph.SPH_FLAG_SYNC), stream)
        s["ctx"] = sph.Context(_params(case, L), stream)
        if kind == "sphenix":
            s["x"] = sph.sph_sphenix_default_params()
            s["av"], s["ac"] = _sphenix_start(seed, n)
            s["out"].update(alpha_v=s["av"], alpha_c=s["ac"])
            sph.sph_step_sphenix(first, s["pool"], s["x"], s["av"], s["ac"])
        else:
            sph.sph_step(first, s["pool"])
        first.close()
        if case["gas"] == "lattices":
            # the step captured in a CUDA graph; the context's scratch is taken up front
            sph.sph_reserve(s["ctx"], n, sims)
            sph.sph_step(s["ctx"], s["pool"])
            torch.cuda.synchronize()
            s["graph"] = torch.cuda.CUDAGraph()
            with torch.cuda.graph(s["graph"], stream=stream):
                sph.sph_step(s["ctx"], s["pool"])
        return s
    if kind == "fof":
        s["ctx"], s["p"] = sph.Context(_params(case, L)), p
        s["b"] = 0.2 * L / n ** (1 / 3)
        s["group"] = torch.empty(n, dtype=torch.int32, device="cuda")
        return s
    d, f = sph.alloc_density(n, n_iter=False), sph.alloc_force(n)
    s.update(ctx=sph.Context(_params(case, L)), p=p, part=sph.particles(p), h=p["h0"], out={**d, **f},
             dens=sph.density_out(d), force=sph.force_out(f))
    if case["nested"] or kind == "masked":
        # what the previous step left: the converged smoothing lengths, off by what a step changes
        for _ in range(12):
            cells = sph.sph_build_cells(s["ctx"], p["x"], p["y"], p["z"], s["h"])
            sph.sph_density(s["ctx"], cells, s["part"], s["h"], s["dens"])
            if not sph.sph_status(s["ctx"]) & sph.SPH_ST_REBUILD:
                break
            s["h"] = d["h"].clone()
        sph.sph_force(s["ctx"], cells, s["part"], s["dens"], s["force"])
        s["h"] = (d["h"] * (1 + 0.002 * (2 * _uni(_gen(seed, 998), n) - 1))).float()
    if kind == "masked":
        s["on"] = _active(case, p)
    return s


def run(s):
    kind = s["case"]["kind"]
    if kind == "step":
        sph.sph_step(s["ctx"], s["pool"])
        return s["out"]
    if kind == "pool":
        if "graph" in s:
            s["graph"].replay()
        else:
            s["out"]["v_sig"].zero_()  # dt = 0: the evaluation alone, at the current state
            sph.sph_step(s["ctx"], s["pool"])
        return s["out"]
    if kind == "sphenix":
        sph.sph_step_sphenix(s["ctx"], s["pool"], s["x"], s["av"], s["ac"])
        return s["out"]
    p, ctx = s["p"], s["ctx"]
    if kind == "fof":
        return sph.sph_fof(ctx, p["x"], p["y"], p["z"], s["b"], s["group"])
    cells = sph.sph_build_cells(ctx, p["x"], p["y"], p["z"], s["h"])
    if kind == "masked":
        sph.sph_density_active(ctx, cells, s["part"], s["h"], s["on"], s["dens"])
        sph.sph_force_active(ctx, cells, s["part"], s["dens"], s["on"], s["force"])
    else:
        sph.sph_density(ctx, cells, s["part"], s["h"], s["dens"])
        sph.sph_force(ctx, cells, s["part"], s["dens"], s["force"])
    return s["out"]


def work(case):
    """Bytes: every input and output array once.  Operations: 33 per density pair of one Newton pass, 66
    of the final pass, 72 per force pair (each add, multiply, divide and root counts one); 4/3 as many
    force pairs as density pairs where supports vary, as larger neighbours reach further."""
    n = sum(nb for _, nb in _box_sizes(case)) if case["kind"] == "pool" else case["n"]
    if case["kind"] == "fof":
        return {"bytes": 28.0 * n, "flops": 0.0}
    ngb = 4 * math.pi / 3 * (GAMMA_K[case["kernel"]] * ETA) ** 3
    per = ngb * (33 + 66) + ngb * (4 / 3 if case["nested"] else 1) * 72
    nbytes = 24 + 20 + 4 + 32 + 20  # positions; v, m, u; h; density results; force results
    if case["kind"] != "loops" and case["kind"] != "masked":
        nbytes += 24 + 16 + 20 + 4  # positions, v, u written back; a, du/dt, v_sig and div v read
    if case["kind"] == "sphenix":
        nbytes, per = nbytes + 16, per + ngb * (30 + 22)  # the gradient pass and the conduction term
    if case["kind"] == "masked":
        per, nbytes = per * case["share"], 24 + 20 + 4 + 1 + 52 * case["share"]
    return {"bytes": float(nbytes) * n, "flops": per * n}


# ---- the same in 64 bits, from the equations ----------------------------------

def _w_dw(q, kernel):
    """w(q) and w'(q) of the kernel (support 1)."""
    pos = lambda v: torch.clamp(v, min=0.0)  # noqa: E731
    a = pos(1 - q)
    if kernel == 0:
        b = pos(0.5 - q)
        return 16 / math.pi * (a ** 3 - 4 * b ** 3), 16 / math.pi * (-3 * a ** 2 + 12 * b ** 2)
    if kernel == 1:
        c, b, d = 15625 / (512 * math.pi), pos(0.6 - q), pos(0.2 - q)
        return c * (a ** 4 - 5 * b ** 4 + 10 * d ** 4), -4 * c * (a ** 3 - 5 * b ** 3 + 10 * d ** 3)
    c = 21 / (2 * math.pi)
    return c * a ** 4 * (1 + 4 * q), -20 * c * q * a ** 3


def _pairs_within(pos, L, sim, t, R):
    """Pairs (i, j, x_i - x_j) with |x_i - x_j| < R_i for the targets t (self included): targets of
    like R share a hash grid of cells that wide; the 27 cells around a target, some 16M candidates at a time."""
    got = []
    order = torch.argsort(R)
    t, R = t[order], R[order]
    at, n = 0, pos.shape[1]
    sim = torch.zeros(n, dtype=torch.int64, device="cuda") if sim is None else sim
    while at < t.shape[0]:
        top = float(R[at]) * 1.26
        end = int(torch.searchsorted(R, torch.tensor(top, dtype=R.dtype, device="cuda")))
        end = max(end, at + 1)
        nc = max(1, min(int(L / float(R[end - 1]) / 1.0000001), 1 << 16))
        c = torch.clamp((pos * (nc / L)).long(), 0, nc - 1)
        key, rank = torch.sort(((sim * nc + c[2]) * nc + c[1]) * nc + c[0])
        tt, RR = t[at:end], R[at:end]
        at = end
        steps = [-1, 0, 1] if nc >= 3 else list(range(nc))
        near = [[torch.remainder(c[k][tt] + o, nc) if nc >= 3 else torch.full_like(tt, o) for o in steps] for k in range(3)]
        ids = torch.stack([((sim[tt] * nc + z) * nc + y) * nc + x for z in near[2] for y in near[1] for x in near[0]], 1)
        lo = torch.searchsorted(key, ids)
        ln = torch.searchsorted(key, ids, right=True) - lo
        cum = torch.cumsum(ln.sum(1), 0)
        k0 = 0
        while k0 < tt.shape[0]:
            done = int(cum[k0 - 1]) if k0 else 0
            k1 = max(k0 + 1, int(torch.searchsorted(cum, done + 16000000, right=True)))
            l, b = ln[k0:k1].reshape(-1), lo[k0:k1].reshape(-1)
            row = torch.repeat_interleave(l)
            j = rank[b[row] + torch.arange(row.shape[0], device="cuda") - (torch.cumsum(l, 0) - l)[row]]
            i = k0 + row // ids.shape[1]
            d = pos[:, tt[i]] - pos[:, j]
            d = d - L * torch.round(d / L)
            keep = (d * d).sum(0) < RR[i] ** 2
            got.append((tt[i[keep]].int(), j[keep].int(), d[:, keep]))
            k0 = k1
    return [torch.cat([v[k] for v in got], -1) for k in range(3)]


class _Gas:
    """Density, gradient and force sums of particles `p` (64 bits) in boxes of side L."""

    def __init__(self, p, h0, L, sim, kernel):
        self.p, self.L, self.kernel, self.n = p, L, kernel, h0.shape[0]
        self.gk = GAMMA_K[kernel]
        pos = torch.stack([p[k] for k in POS])
        n, gk, dev = self.n, self.gk, "cuda"
        h = torch.zeros(n, dtype=torch.float64, device=dev)
        target = (gk * ETA) ** 3
        todo, R = torch.arange(n, device=dev), 1.02 * gk * h0.double()
        kept = []
        for _ in range(60):
            i, j, d = _pairs_within(pos, L, sim, todo, R)
            r = d.square().sum(0).sqrt()
            Rn = torch.zeros(n, dtype=torch.float64, device=dev)
            Rn[todo] = R
            # the root of sum_j w(r/H) = (gamma_K eta)^3, which lies within R where the sum at R reaches it
            ok = self._add(_w_dw(r / Rn[i.long()], kernel)[0], i) >= target
            lo, hi, H = torch.zeros_like(Rn), Rn.clone(), torch.where(ok, 0.97 * Rn, torch.ones_like(Rn))
            mine = ok[i.long()]
            i, j, d, r = i[mine], j[mine], d[:, mine], r[mine]
            il = i.long()
            for _ in range(100):
                q = r / H[il]
                w, dw = _w_dw(q, kernel)
                S, dS = self._add(w, i), self._add(-dw * q, i)  # dS: H dS/dH
                hi, lo = torch.where(S >= target, H, hi), torch.where(S < target, H, lo)
                new = H * (1 - (S - target) / torch.clamp(dS, min=1e-30))
                new = torch.where((new >= lo) & (new <= hi), new, 0.5 * (lo + hi))
                new = torch.where(ok, new, H)
                off = float((new / H - 1).abs().max())
                H = new
                if off < 1e-13:
                    break
            h[ok] = H[ok] / gk
            near = r < H[il]
            kept.append((i[near], j[near], d[:, near]))
            left = ~ok[todo]
            todo, R = todo[left], R[left] * 1.2
            if todo.shape[0] == 0:
                break
        self.i, self.j, d = [torch.cat([v[k] for v in kept], -1) for k in range(3)]
        other = self.i != self.j
        self.h, self.H = h, gk * h
        # density sums over the pairs of each particle's support, itself included
        i, j, d, m = self.i.long(), self.j.long(), d, p["m"]
        r = d.square().sum(0).sqrt()
        q = r / self.H[i]
        w, dw = _w_dw(q, kernel)
        H3 = self.H ** 3
        o = self.out = {"h": h}
        rho = o["rho"] = self._add(m[j] * w, i) / H3
        drho = -self._add(m[j] * (3 * w + q * dw), i) / (h * H3)
        o["f"] = 1 / (1 + h / (3 * rho) * drho)
        G = torch.where(r > 0, dw / torch.clamp(r, min=1e-300), torch.zeros_like(r)) / self.H[i] ** 4
        v = [p[k][i] - p[k][j] for k in ("vx", "vy", "vz")]
        mg = m[j] * G
        o["div_v"] = -self._add(mg * (v[0] * d[0] + v[1] * d[1] + v[2] * d[2]), i) / rho
        curl = [self._add(mg * (v[a] * d[b] - v[b] * d[a]), i) / rho for a, b in ((1, 2), (2, 0), (0, 1))]
        o["curl_v"] = torch.sqrt(sum(k * k for k in curl))
        o["P"] = (GAMMA - 1) * p["u"] * rho
        o["c"] = torch.sqrt(GAMMA * o["P"] / rho)
        o["balsara"] = o["div_v"].abs() / (o["div_v"].abs() + o["curl_v"] + EPS_B * o["c"] / h)
        del v, G, mg, w, dw, q
        self.i, self.j, self.d, self.r = self.i[other], self.j[other], d[:, other], r[other]

    def _add(self, v, i):
        return torch.zeros(self.n, dtype=torch.float64, device="cuda").index_add_(0, i.long(), v)

    def _most(self, v, i, start=None):
        out = torch.zeros(self.n, dtype=torch.float64, device="cuda") if start is None else start.clone()
        return out.scatter_reduce_(0, i.long(), v, "amax")

    def _grad(self, r, H):
        return _w_dw(r / H, self.kernel)[1] / r / H ** 4

    def _v_cond(self, i, j, vx, r):
        o = self.out
        return vx.abs() / r + torch.sqrt(2 * (o["P"][i] - o["P"][j]).abs() / (o["rho"][i] + o["rho"][j]))

    def gradient(self, av, ac, dt):
        """The SPHENIX conduction parameter after dt (ell, beta_c and the limits at their defaults)."""
        p, o, i, j = self.p, self.out, self.i.long(), self.j.long()
        vx = sum((p["v" + k][i] - p["v" + k][j]) * self.d[n] for n, k in enumerate(POS))
        lap = 2 * self._add(p["m"][j] / o["rho"][j] * (p["u"][i] - p["u"][j]) * self._grad(self.r, self.H[i]), i)
        vc = self._most(self._v_cond(i, j, vx, self.r), i)
        most = self._most(av[j], i, av)
        new = ac + dt * (self.H * lap / torch.sqrt(p["u"]) - ac * vc / self.H)
        return torch.clamp(torch.minimum(new, 1 - most / 2), min=0.0)

    def force(self, av=None, ac=None):
        """Force sums over the pairs with r < max(H_i, H_j): a pair within H_i alone counts for j as well."""
        p, o, n = self.p, self.out, self.n
        rev = self.r >= self.H[self.j.long()]
        out = {k: torch.zeros(n, dtype=torch.float64, device="cuda") for k in sph.FORCE_FIELDS}
        for i, j, d, r in ((self.i, self.j, self.d, self.r), (self.j[rev], self.i[rev], -self.d[:, rev], self.r[rev])):
            for k0 in range(0, i.shape[0], 1 << 25):
                part = slice(k0, k0 + (1 << 25))
                ii, jj, dd, rr = i[part].long(), j[part].long(), d[:, part], r[part]
                vx = sum((p["v" + k][ii] - p["v" + k][jj]) * dd[a] for a, k in enumerate(POS))
                Gi, Gj = self._grad(rr, self.H[ii]), self._grad(rr, self.H[jj])
                mu, rs = torch.clamp(vx, max=0.0) / rr, o["rho"][ii] + o["rho"][jj]
                vs = o["c"][ii] + o["c"][jj] - BETA_V * mu
                alpha = (ALPHA_V if av is None else 0.5 * (av[ii] + av[jj])) * 0.5 * (o["balsara"][ii] + o["balsara"][jj])
                nu = -alpha * mu * vs / (0.5 * rs)
                pi = o["f"][ii] * o["P"][ii] / o["rho"][ii] ** 2 * Gi
                pj = o["f"][jj] * o["P"][jj] / o["rho"][jj] ** 2 * Gj
                visc, m = o["f"][ii] * Gi + o["f"][jj] * Gj, p["m"][jj]
                s = m * (pi + pj + 0.5 * nu * visc)
                for a, k in enumerate(("ax", "ay", "az")):
                    out[k].index_add_(0, ii, -s * dd[a])
                du = m * (pi + 0.25 * nu * visc) * vx
                if av is not None:
                    Pi, Pj = o["P"][ii], o["P"][jj]
                    acij = (Pi * ac[ii] + Pj * ac[jj]) / (Pi + Pj)
                    du = du + acij * self._v_cond(ii, jj, vx, rr) * m * (p["u"][ii] - p["u"][jj]) * visc * rr / rs
                out["du_dt"].index_add_(0, ii, du)
                out["v_sig"].scatter_reduce_(0, ii, vs, "amax")
        return out


def exact(case, seed):
    if case["kind"] == "fof":
        return None
    p, L, sim, off = _inputs(case, seed)
    h0, n, kind = p.pop("h0"), p["x"].shape[0], case["kind"]
    p = {k: v.double() for k, v in p.items()}
    G = _Gas(p, h0, L, sim, case["kernel"])
    av, ac = (v.double() for v in _sphenix_start(seed, n)) if kind == "sphenix" else (None, None)
    if av is not None:
        # no signal velocity yet, and dt = 0: convergence alone drives nothing
        ac = G.gradient(av, ac, 0.0)
    o = {**G.out, **G.force(av, ac)}
    if kind in ("loops", "masked"):
        return o
    steps = {"lattices": 2, "boxes": 0}.get(case["gas"], 1)  # a captured step had a plain one before it
    sims = torch.zeros(n, dtype=torch.int64, device="cuda") if sim is None else sim
    for _ in range(steps):
        q = torch.full((off.shape[0] - 1,), math.inf, dtype=torch.float64, device="cuda")
        dt = CFL * G.gk * q.scatter_reduce_(0, sims, o["h"] / o["v_sig"], "amin")[sims]
        rate = {"vx": o["ax"], "vy": o["ay"], "vz": o["az"], "u": o["du_dt"]}
        half = {k: p[k] + 0.5 * dt * rate[k] for k in rate}
        new = {k: torch.remainder(p[k] + dt * half["v" + k], L) for k in POS}
        G = _Gas({**new, **{k: half[k] + 0.5 * dt * rate[k] for k in rate}, "m": p["m"]}, o["h"], L, sim, case["kernel"])
        if av is not None:
            S = G.H ** 2 * torch.clamp(-(G.out["div_v"] - o["div_v"]) / dt, min=0.0)
            loc = 2 * S / (o["v_sig"] ** 2 + S)
            av = torch.where(loc > av, loc, loc + (av - loc) * torch.exp(-0.05 * G.out["c"] * dt / G.H))
            ac = G.gradient(av, ac, dt)
        o = {**G.out, **G.force(av, ac)}
        rate = {"vx": o["ax"], "vy": o["ay"], "vz": o["az"], "u": o["du_dt"]}
        p = {**new, **{k: half[k] + 0.5 * dt * rate[k] for k in rate}, "m": p["m"]}
    o.update({k: p[k] for k in POS + ("vx", "vy", "vz", "u")})
    return {**o, "alpha_v": av, "alpha_c": ac} if av is not None else o
