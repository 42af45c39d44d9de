"""Timed workloads of the DPDE step: what a simulation program has the library do.

A pass hands the library a state, advances it and takes the new state back
(``dpde_set_state``, ``dpde_step`` and ``dpde_get_state`` through
:class:`~paper_1507_06643_gb300.dpde.System`), or reads the observables of the
state it holds. A program keeps its handle from pass to pass, so the handle is
made in :func:`prepare`; states stay on the GPU (torch tensors), except in the
two small cases, whose programs hold numpy arrays.

A case is a dict of
  family     fluid | shock | batch | lj   -- how the particles are laid out
  op         step | observables
  scheme     SER | HYBRID | SEM | SSA
  precision  mixed | fp64
  n, density, cv, kT, sigma, dt, steps
  bx, by, bz       Hybrid domains per axis (one replica)
  fx, fy, fz       box edges relative to each other
  reps, n_max, sizes_seed   (batch) replica sizes log-uniform in [n, n_max]
  start      uniform | relaxed -- independent uniform positions, as a run
             begins, or one particle per site of a jittered grid, whose number
             fluctuations are those of a fluid under repulsion
  walls      (shock) closed along z by a fixed wall and a piston
  project    the projection on the internal energies is on
  host       states are numpy arrays on the host
"""
import math
import random

import numpy as np
import torch

from paper_1507_06643_gb300 import dpde

A_SOFT = 25.0          # soft-repulsion amplitude of every soft fluid
SHOCK_SPEED = 2.0      # velocity of the two halves of a shock run
SHOCK_FACTOR = 1.57    # density behind the front, over the density ahead of it
RAREFIED = 0.6         # density behind the expansion at the other end


# ---- the cases -------------------------------------------------------------------------

def _case(name, family, scheme, precision, n, **kw):
    c = dict(name=name, family=family, op="step", scheme=scheme, precision=precision, n=n, density=3.0, cv=100.0,
             kT=1.0, sigma=3.0, dt=0.01, steps=5, bx=1, by=1, bz=1, fx=1.0, fy=1.0, fz=1.0, reps=1, n_max=0,
             sizes_seed=0, start="relaxed", walls=False, project=False, host=False)
    c.update(kw)
    return c


def listed():
    return [
        # the smallest call: a method study's box in double precision, launch and latency bound
        _case("plain_hybrid_fp64", "fluid", "HYBRID", "fp64", 1000, bx=2, by=2, bz=2, steps=10, start="uniform",
              host=True),
        # a few independent trajectories of the paper's N = 343 Lennard-Jones system, sequential scheme
        _case("trajectories_lj_ssa", "lj", "SSA", "mixed", 343, density=0.8095, sigma=2.0, dt=0.002, steps=10, reps=16,
              n_max=343, host=True),
        # the equilibrium fluid, a simulation of ordinary size
        _case("equilibrium_hybrid", "fluid", "HYBRID", "mixed", 108000, bx=5, by=5, bz=5, steps=10),
        # its double-precision control run, with the projection that pins the total energy
        _case("equilibrium_hybrid_fp64", "fluid", "HYBRID", "fp64", 108000, bx=5, by=5, bz=5, steps=2, project=True),
        # the fully parallel scheme: every pair through the two sweeps
        _case("fluid_ser", "fluid", "SER", "mixed", 1000000, cv=50.0, steps=4),
        # Euler-Maruyama on an oblong box of odd size
        _case("oblong_sem", "fluid", "SEM", "mixed", 250047, fx=2.0, fy=1.0, fz=0.5, steps=5),
        # the sequential scheme over one whole replica
        _case("whole_ssa", "fluid", "SSA", "mixed", 64000, steps=4),
        # the paper's Lennard-Jones fluid: long neighbour lists
        _case("lj_hybrid", "lj", "HYBRID", "mixed", 144000, density=0.8095, cv=10.0, sigma=2.0, dt=0.002, bx=5, by=5,
              bz=5, steps=4),
        # the large fluid, just started: the throughput benchmark
        _case("large_hybrid", "fluid", "HYBRID", "mixed", 4000000, cv=50.0, bx=18, by=18, bz=18, steps=5,
              start="uniform"),
        # the shock tube some way into its run: a compressed and a rarefied slab
        _case("shock_hybrid", "shock", "HYBRID", "mixed", 3840000, dt=0.005, bx=8, by=8, bz=160, fz=20.0, steps=5),
        # many independent systems of uneven size and temperature in one handle
        _case("batched_hybrid", "batch", "HYBRID", "mixed", 2000, cv=0.0, kT=0.0, reps=256, n_max=64000,
              sizes_seed=1005, steps=5),
        # what a run samples between steps
        _case("fluid_observables", "fluid", "SER", "mixed", 1000000, cv=50.0, op="observables", steps=0),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _bricks(c, per_domain):
    """Hybrid domains of about `per_domain` particles, each at least one cell wide and three cells in the box."""
    rc = _r_cut(c)
    for a, edge in zip("xyz", _box(c, c["n"])):
        domain = (per_domain / c["density"]) ** (1.0 / 3.0)
        b = max(1, min(int(round(edge / domain)), int(edge / rc)))
        while b > 1 and b * int(edge / (b * rc)) < 3:
            b -= 1
        c["b" + a] = b


def draw(rng):
    """One more case. Particle counts run over the listed range on a logarithmic scale; the steps of a pass
    keep its work within the largest listed one's."""
    kind = rng.choice(["hybrid", "hybrid", "hybrid_fp64", "ser", "sem", "ssa", "lj", "lj_traj", "shock", "batch",
                       "observables"])
    density = rng.uniform(2.5, 3.5)
    cv = rng.choice([10.0, 50.0, 100.0])
    if kind == "hybrid":
        c = _case("", "fluid", "HYBRID", "mixed", _log_int(rng, 1000, 4000000), density=density, cv=cv,
                  start=rng.choice(["uniform", "relaxed"]), fy=rng.uniform(0.6, 1.0), fz=rng.uniform(0.6, 1.0))
        c["steps"] = max(1, min(10, 20000000 // c["n"]))
        _bricks(c, rng.uniform(300.0, 1800.0))
    elif kind == "hybrid_fp64":
        c = _case("", "fluid", "HYBRID", "fp64", _log_int(rng, 1000, 110000), density=density, cv=cv,
                  project=rng.random() < 0.5, steps=rng.randint(1, 2))
        _bricks(c, rng.uniform(300.0, 1200.0))
    elif kind in ("ser", "sem"):
        c = _case("", "fluid", kind.upper(), rng.choice(["mixed", "mixed", "fp64"]), _log_int(rng, 1000, 1000000),
                  density=density, cv=cv, fx=rng.uniform(0.7, 1.5), fz=rng.uniform(0.7, 1.5))
        if c["precision"] == "fp64":
            c["n"] = min(c["n"], 150000 + c["n"] % 1000)
        c["steps"] = max(1, min(8, 4000000 // c["n"])) if c["precision"] == "mixed" else 1
    elif kind == "ssa":
        c = _case("", "fluid", "SSA", "mixed", _log_int(rng, 1000, 200000), density=density, cv=cv)
        c["steps"] = rng.randint(1, 4)
    elif kind == "lj":
        c = _case("", "lj", rng.choice(["HYBRID", "SER"]), "mixed", _log_int(rng, 2000, 144000), density=0.8095,
                  cv=rng.choice([10.0, 50.0]), sigma=2.0, dt=0.002, steps=rng.randint(1, 4))
        _bricks(c, rng.uniform(500.0, 2000.0))
    elif kind == "lj_traj":
        c = _case("", "lj", rng.choice(["SSA", "SER"]), "mixed", 343, density=0.8095, sigma=2.0, dt=0.002,
                  steps=rng.randint(3, 10), reps=rng.randint(4, 32), n_max=rng.choice([343, 1000]),
                  sizes_seed=rng.randint(1, 1 << 30), host=True)
    elif kind == "shock":
        c = _case("", "shock", "HYBRID", "mixed", _log_int(rng, 60000, 3840000), density=density, cv=cv, dt=0.005,
                  fz=rng.uniform(6.0, 20.0), walls=rng.random() < 0.3)
        c["steps"] = max(1, min(8, 19000000 // c["n"]))
        _bricks(c, rng.uniform(350.0, 1000.0))
    elif kind == "batch":
        c = _case("", "batch", "HYBRID", "mixed", 2000, density=density, cv=0.0, kT=0.0, reps=rng.randint(8, 256),
                  n_max=_log_int(rng, 8000, 64000), sizes_seed=rng.randint(1, 1 << 30), steps=rng.randint(1, 5))
    else:
        c = _case("", "fluid", "SER", rng.choice(["mixed", "mixed", "fp64"]), _log_int(rng, 1000, 1000000),
                  density=density, cv=cv, op="observables", steps=0, start=rng.choice(["uniform", "relaxed"]))
        if c["precision"] == "fp64":
            c["n"] = min(c["n"], 150000 + c["n"] % 1000)
    del c["name"]
    return c


# ---- the systems of a case ---------------------------------------------------------------

def _r_cut(c):
    return 2.5 if c["family"] == "lj" else 1.0


def _box(c, n):
    f = (c["fx"], c["fy"], c["fz"])
    s = (n / c["density"] / (f[0] * f[1] * f[2])) ** (1.0 / 3.0)
    return tuple(s * x for x in f)


def _replicas(c):
    """(n, box, C_v, kT, domains) of every replica."""
    one = (c["n"], _box(c, c["n"]), c["cv"], c["kT"], (c["bx"], c["by"], c["bz"]))
    if c["reps"] == 1:
        return [one]
    rng = random.Random(c["sizes_seed"])
    out = []
    for _ in range(c["reps"]):
        n = _log_int(rng, c["n"], c["n_max"]) if c["n_max"] > c["n"] else c["n"]
        box = _box(c, n)
        b = max(1, int(round((n / 1000.0) ** (1.0 / 3.0)))) if c["scheme"] == "HYBRID" else 1
        while b > 1 and b * int(box[0] / (b * _r_cut(c))) < 3:
            b -= 1
        out.append((n, box, c["cv"] or rng.choice([10.0, 50.0, 100.0]), c["kT"] or rng.uniform(0.5, 2.0), (b, b, b)))
    return out


def _params(c, seed):
    lj = c["family"] == "lj"
    return dpde.make_params(mass=1.0, r_cut=_r_cut(c), a=A_SOFT, sigma=c["sigma"], seed=1000 + seed,
                            precision=c["precision"], potential=dpde.POT_LJ if lj else dpde.POT_SOFT)


def _shock_profile(c, u):
    """Position along z (of the box edge) and velocity at the mass fraction u of a shock run."""
    if c["walls"]:       # everything moves down on the wall at z = 0; the slab there has stopped
        seg = [(0.25, SHOCK_FACTOR, 0.0), (0.75, 1.0, -SHOCK_SPEED)]
    else:                # halves collide at the middle and part at the periodic end
        a = 0.15
        b = a * (SHOCK_FACTOR - 1.0) / (1.0 - RAREFIED)
        free = 0.5 - a - b
        seg = [(b, RAREFIED, 0.0), (free, 1.0, SHOCK_SPEED), (2 * a, SHOCK_FACTOR, 0.0), (free, 1.0, -SHOCK_SPEED),
               (b, RAREFIED, 0.0)]
    mass = [w * f for w, f, _ in seg]
    z, v, m0, z0 = torch.zeros_like(u), torch.zeros_like(u), 0.0, 0.0
    for (w, _, vel), m in zip(seg, mass):
        f0, f1 = m0 / sum(mass), (m0 + m) / sum(mass)
        here = (u >= f0) & (u < f1)
        z = torch.where(here, z0 + w * (u - f0) / (f1 - f0), z)
        v = torch.where(here, torch.full_like(v, vel), v)
        m0, z0 = m0 + m, z0 + w
    return z, v


def _sites(gen, n, box, jitter, dev):
    """n points in the box, each jittered about a site of its own of a grid."""
    h = (box[0] * box[1] * box[2] / n) ** (1.0 / 3.0)
    g = [max(1, int(round(b / h))) for b in box]
    while g[0] * g[1] * g[2] < n:
        k = max(range(3), key=lambda a: box[a] / g[a])
        g[k] += 1
    s = torch.randperm(g[0] * g[1] * g[2], generator=gen, device=dev)[:n]
    site = torch.stack([s % g[0], (s // g[0]) % g[1], s // (g[0] * g[1])], 1).double()
    site += 0.5 + jitter * (torch.rand(n, 3, generator=gen, device=dev, dtype=torch.float64) - 0.5)
    edge = torch.tensor([b / k for b, k in zip(box, g)], dtype=torch.float64, device=dev)
    return site * edge


def _state(c, seed, dev):
    """(q, p, eps) of all replicas: positions by the case's layout, Maxwellian momenta without drift,
    internal energies C_v kT with a 5 % spread."""
    gen = torch.Generator(device=dev).manual_seed(seed * 2654435761 % (1 << 62) + 17)
    qs, ps, es = [], [], []
    for n, box, cv, kT, _ in _replicas(c):
        L = torch.tensor(box, dtype=torch.float64, device=dev)
        if c["start"] == "uniform":
            q = torch.rand(n, 3, generator=gen, device=dev, dtype=torch.float64) * L
        else:
            q = _sites(gen, n, box, 0.2 if c["family"] == "lj" else 0.9, dev)
        p = torch.randn(n, 3, generator=gen, device=dev, dtype=torch.float64) * math.sqrt(kT)
        if c["op"] == "step":   # (a total momentum of zero would be sampled as rounding alone)
            p -= p.mean(0, keepdim=True)
        if c["family"] == "shock":
            z, v = _shock_profile(c, (q[:, 2] / L[2]).clamp(0.0, 1.0 - 1e-12))
            q[:, 2] = z * L[2]
            p[:, 2] += v
        e = cv * kT * (1.0 + 0.05 * (2.0 * torch.rand(n, generator=gen, device=dev, dtype=torch.float64) - 1.0))
        qs.append(torch.where(q >= L, torch.zeros_like(q), q))
        ps.append(p)
        es.append(e)
    return torch.cat(qs).contiguous(), torch.cat(ps).contiguous(), torch.cat(es).contiguous()


# ---- a pass --------------------------------------------------------------------------------

def prepare(case, seed):
    c = case
    dev = torch.device("cuda")
    q, p, e = _state(c, seed, dev)
    walls = (1, -SHOCK_SPEED) if c["walls"] else (0, 0.0)
    S = dpde.System(_params(c, seed), [dpde.make_replica(n, box, cv, br, *walls) for n, box, cv, _, br in _replicas(c)])
    torch.cuda.synchronize()
    st = {"S": S, "case": c}
    if c["host"]:
        st["in"] = tuple(x.cpu().numpy() for x in (q, p, e))
    else:
        st["in"] = (q, p, e)
        st["out"] = tuple(torch.empty_like(x) for x in (q, p, e))
    if c["project"] or c["op"] == "observables":
        S.set_state(*st["in"], on_device=not c["host"])
    if c["project"]:
        S.set_projection(True)
    return st


def run(state):
    S, c = state["S"], state["case"]
    if c["op"] == "observables":
        return S.observables(check=True)
    S.set_state(*state["in"], on_device=not c["host"])
    S.step(c["steps"], c["dt"], c["scheme"])
    if c["host"]:
        q, p, e = S.get_state()
    else:
        q, p, e = state["out"]
        rc = dpde.dpde_get_state(S.h, q, p, e, on_device=True)
        if rc != dpde.DPDE_OK:
            raise RuntimeError(f"dpde_get_state: status {rc}")
    return {"q": q, "p": p, "eps": e}


def work(case):
    c = case
    reps = _replicas(c)
    n = sum(r[0] for r in reps)
    pairs = n * 2.0 / 3.0 * math.pi * c["density"] * _r_cut(c) ** 3
    word = 8 if c["precision"] == "fp64" else 4
    if c["op"] == "observables":
        # the state read once; per pair the distance, the potential and its Laplacian
        return {"bytes": n * (9 * word + 8), "flops": 25.0 * pairs}
    # 7 doubles in and out per particle; per step and pair the force, the pair's Gaussians and the map
    # (or the two sweeps' arithmetic)
    return {"bytes": 2 * 56 * n, "flops": c["steps"] * pairs * (20.0 + 180.0 + 95.0)}


# ---- the same in 64 bits, from the paper's equations ----------------------------------------

def _neighbours(q, L, rc, per):
    """Pairs (i, j, q_i - q_j) within rc, each once, from cells at least rc wide; per: periodic axes."""
    dev, n = q.device, len(q)
    nc = [max(3, int(L[a] / rc)) for a in range(3)]
    Lt = torch.tensor(L, dtype=torch.float64, device=dev)
    nct = torch.tensor(nc, device=dev)
    c = torch.minimum((q * (nct / Lt)).long().clamp_(min=0), nct - 1)
    lin = (c[:, 2] * nc[1] + c[:, 1]) * nc[0] + c[:, 0]
    order = torch.argsort(lin, stable=True)
    cells = nc[0] * nc[1] * nc[2]
    count = torch.bincount(lin, minlength=cells)
    first = torch.cumsum(count, 0) - count
    M = int(count.max())
    table = torch.full((cells, M), -1, dtype=torch.long, device=dev)
    table[lin[order], torch.arange(n, device=dev) - first[lin[order]]] = order
    idx = torch.arange(cells, device=dev)
    cx, cy, cz = idx % nc[0], (idx // nc[0]) % nc[1], idx // (nc[0] * nc[1])
    got = []
    step = max(1, 20000000 // (M * M))
    for off in [(0, 0, 0)] + [(x, y, z) for z in (0, 1) for y in (-1, 0, 1) for x in (-1, 0, 1)
                              if (z, y, x) > (0, 0, 0)]:
        x, y, z = cx + off[0], cy + off[1], cz + off[2]
        ok = torch.ones_like(idx, dtype=torch.bool)
        for a, v in enumerate((x, y, z)):
            if not per[a]:
                ok &= (v >= 0) & (v < nc[a])
        other = ((z % nc[2]) * nc[1] + y % nc[1]) * nc[0] + x % nc[0]
        for s in range(0, cells, step):
            here = idx[s:s + step][ok[s:s + step]]
            ti, tj = table[here], table[other[here]]
            i = ti[:, :, None].expand(-1, -1, M).reshape(-1)
            j = tj[:, None, :].expand(-1, M, -1).reshape(-1)
            keep = (i >= 0) & (j >= 0)
            if off == (0, 0, 0):
                keep &= i < j
            i, j = i[keep], j[keep]
            d = q[i] - q[j]
            for a in range(3):
                if per[a]:
                    d[:, a] -= L[a] * torch.round(d[:, a] / L[a])
            near = (d * d).sum(1) < rc * rc
            got.append((i[near], j[near], d[near]))
    return tuple(torch.cat([g[k] for g in got]) for k in range(3))


def _potential(c, r):
    """v(r), -v'(r)/r and v'' + 2 v'/r."""
    rc = _r_cut(c)
    if c["family"] != "lj":
        w = 1.0 - r / rc
        return 0.5 * A_SOFT * rc * w * w, A_SOFT * w / r, A_SOFT / rc - 2.0 * A_SOFT * w / r
    k6 = rc ** -6.0
    shift, slope = 4.0 * (k6 * k6 - k6), 4.0 * (6.0 * k6 - 12.0 * k6 * k6) / rc
    s6 = r ** -6.0
    dv = 4.0 * (6.0 * s6 - 12.0 * s6 * s6) / r - slope
    v = 4.0 * (s6 * s6 - s6) - shift - slope * (r - rc)
    return v, -dv / r, 4.0 * (156.0 * s6 * s6 - 42.0 * s6) / (r * r) + 2.0 * dv / r


def _gauss(seed, step, rep, i, j):
    """The noise of pairs (i, j): Philox4x32-10 (Salmon et al., SC'11) on the ordered ids, Box-Muller."""
    m32 = 0xFFFFFFFF
    x0, x1 = torch.minimum(i, j), torch.maximum(i, j)
    x2, x3 = torch.full_like(i, step), torch.full_like(i, rep)
    k0, k1 = seed & m32, seed >> 32
    for r in range(10):
        p0, p1 = x0 * 0xD2511F53, x2 * 0xCD9E8D57       # modulo 2^64: the bits of the full product
        x0, x1, x2, x3 = ((p1 >> 32) & m32) ^ x1 ^ k0, p1 & m32, ((p0 >> 32) & m32) ^ x3 ^ k1, p0 & m32
        k0, k1 = (k0 + 0x9E3779B9) & m32, (k1 + 0xBB67AE85) & m32
    u1, u2 = (((x >> 8) + 1).double() * 2.0 ** -24 for x in (x0, x2))
    t1, t2 = ((x >> 8).double() * (2.0 * math.pi * 2.0 ** -24) for x in (x1, x3))
    r1, r2 = torch.sqrt(-2.0 * torch.log(u1)), torch.sqrt(-2.0 * torch.log(u2))
    g = torch.stack([r1 * torch.cos(t1), r1 * torch.sin(t1), r2 * torch.cos(t2)], 1)
    return torch.where((i < j)[:, None], g, -g)


def _ssa_sequence(c, q, L, per, bricks, i, j):
    """Of the pairs, those inside one domain as (first, second, their index) in sequence order, and whether
    each pair is inside one."""
    rc = _r_cut(c)
    B = (1, 1, 1) if c["scheme"] == "SSA" else bricks
    nc = [bricks[a] * int(L[a] / (bricks[a] * rc)) for a in range(3)]
    k = [nc[a] // B[a] for a in range(3)]
    cell = np.stack([np.minimum(nc[a] - 1, (q[:, a] * (nc[a] / L[a])).astype(np.int64)) for a in range(3)], 1)
    inside = np.all(cell[i] // k == cell[j] // k, axis=1)
    pair = np.nonzero(inside)[0]
    s, t = i[pair], j[pair]
    d = cell[t] - cell[s]
    for a in range(3):
        if per[a]:
            d[:, a] = np.where(d[:, a] > 1, d[:, a] - nc[a], np.where(d[:, a] < -1, d[:, a] + nc[a], d[:, a]))
    seg = 9 * (d[:, 2] + 1) + 3 * (d[:, 1] + 1) + d[:, 0] + 1
    swap = (seg < 13) | ((seg == 13) & (t < s))
    s, t = np.where(swap, t, s), np.where(swap, s, t)
    seg = np.where(swap, 26 - seg, seg)
    colour = np.zeros(len(q), np.int64)
    for a in (2, 1, 0):
        P = 2 if a == 2 else 3
        l = cell[:, a] % k[a]
        full = P * (k[a] // P)
        col = np.where((B[a] == 1) & per[a] & (l >= full), P + l - full, l % P)
        colour = colour * 5 + col
    lin = (cell[:, 2] * nc[1] + cell[:, 1]) * nc[0] + cell[:, 0]
    order = np.lexsort((t, seg, s, lin[s], colour[s]))
    return s[order], t[order], pair[order], inside


def _levels(n, s, t):
    """Level of every map of a sequence: one above the last earlier map of either particle."""
    last = [0] * n
    lev = []
    for a, b in zip(s.tolist(), t.tolist()):
        x = last[a] if last[a] > last[b] else last[b]
        last[a] = last[b] = x + 1
        lev.append(x)
    return np.asarray(lev, np.int64)


def _exact_steps(c, seed, reps, q, p, e):
    """The steps of all replicas, their particles in one index space."""
    per = (True, True, True)
    dt, sigma, rc, scheme = c["dt"], c["sigma"], _r_cut(c), c["scheme"]
    first = np.concatenate([[0], np.cumsum([r[0] for r in reps])]).tolist()
    own = [slice(a, b) for a, b in zip(first[:-1], first[1:])]
    L = torch.cat([torch.tensor(r[1], dtype=torch.float64, device=q.device).expand(r[0], 3) for r in reps])
    cv = torch.cat([torch.full((r[0],), r[2], dtype=torch.float64, device=q.device) for r in reps])

    def forces(q):
        pairs = [_neighbours(q[o], r[1], rc, per) for o, r in zip(own, reps)]
        i, j = (torch.cat([x[k] + o.start for x, o in zip(pairs, own)]) for k in (0, 1))
        d = torch.cat([x[2] for x in pairs])
        r = torch.sqrt((d * d).sum(1))
        v, fr, lap = _potential(c, r)
        F = torch.zeros_like(q)
        F.index_add_(0, i, fr[:, None] * d)
        F.index_add_(0, j, -fr[:, None] * d)
        m = [len(x[0]) for x in pairs]
        return pairs, i, j, 1.0 - r / rc, F, [x.sum() for x in v.split(m)], [2.0 * x.sum() for x in lap.split(m)]

    def energies(U, p, e):
        return [u + 0.5 * (p[o] * p[o]).sum() + e[o].sum() for o, u in zip(own, U)]

    pairs, i, j, w, F, U, lap = forces(q)
    if c["op"] == "observables":
        out = []
        for o, r, u, la in zip(own, reps, U, lap):
            k, eint, mom = 0.5 * (p[o] * p[o]).sum(), e[o].sum(), p[o].sum(0)
            out.append({"E": float(u + k + eint), "K": float(k), "U": float(u), "Eint": float(eint),
                        "Px": float(mom[0]), "Py": float(mom[1]), "Pz": float(mom[2]),
                        "Tkin": float(2 * k / (3 * (r[0] - 1))), "Tint": float(r[0] / (r[2] / e[o]).sum()),
                        "Tpot_num": float((F[o] * F[o]).sum()), "Tpot_den": float(la), "step": 0, "n": r[0],
                        "neg_eps": 0, "nonfinite": 0})
        return out
    E0 = energies(U, p, e)
    for step in range(c["steps"]):
        p = p + 0.5 * dt * F
        q = q + dt * p
        q = torch.where(q >= L, q - L, torch.where(q < 0.0, q + L, q))
        pairs, i, j, w, F, U, _ = forces(q)
        p = p + 0.5 * dt * F
        G = torch.cat([_gauss(1000 + seed, step, k, x[0], x[1]) for k, x in enumerate(pairs)])
        rest = torch.ones(len(i), dtype=torch.bool, device=q.device)
        if scheme in ("SSA", "HYBRID"):
            seq, at = [], 0
            for o, r, x in zip(own, reps, pairs):
                s, t, pair, inside = _ssa_sequence(c, q[o].cpu().numpy(), r[1], per, r[4], x[0].cpu().numpy(),
                                                   x[1].cpu().numpy())
                seq.append((s + o.start, t + o.start, pair + at))
                rest[at:at + len(inside)] = torch.from_numpy(~inside).to(q.device)
                at += len(inside)
            s, t, pair = (np.concatenate([x[k] for x in seq]) for k in range(3))
            lev = _levels(len(q), s, t)
            order = np.argsort(lev, kind="stable")
            cuts = np.searchsorted(lev[order], np.arange(lev.max() + 2 if len(lev) else 1)).tolist()
            s, t, pair = (torch.from_numpy(x[order]).to(q.device) for x in (s, t, pair))
            g = torch.where((i[pair] == s)[:, None], G[pair], -G[pair])
            wp, cs, ct = w[pair], cv[s], cv[t]
            p, e = p.clone(), e.clone()
            for b, f in zip(cuts[:-1], cuts[1:]):
                a, o = s[b:f], t[b:f]
                ps, pt, es, et = p[a], p[o], e[a], e[o]
                gam = 0.25 * sigma * sigma * (cs[b:f] / es + ct[b:f] / et)
                x = 2.0 * gam * wp[b:f] ** 2 * dt
                amp = sigma * torch.sqrt(-torch.expm1(-2.0 * x) / gam)
                D = 0.5 * (torch.expm1(-x)[:, None] * (ps - pt) + amp[:, None] * g[b:f])
                dK = 0.5 * (D * (2.0 * (ps - pt + D))).sum(1)
                p[a], p[o] = ps + D, pt - D
                e[a], e[o] = es - 0.5 * dK, et - 0.5 * dK
        if scheme != "SSA":
            a, o, wr, g = i[rest], j[rest], w[rest], G[rest]
            gam, v, chi = 0.25 * sigma * sigma * (cv[a] / e[a] + cv[o] / e[o]), p[a] - p[o], wr * wr
            noise = (sigma * math.sqrt(dt) * wr)[:, None] * g
            dij = -(gam * chi * dt)[:, None] * v + noise
            dp = torch.zeros_like(p)
            dp.index_add_(0, a, dij)
            dp.index_add_(0, o, -dij)
            if scheme == "SEM":
                de = 0.5 * (gam * (v * v).sum(1) - 3.0 * sigma * sigma) * chi * dt - 0.5 * (v * noise).sum(1)
                e = e.index_add(0, a, de).index_add(0, o, de)
            else:
                T = (dij * (p[a] + p[o] + 0.5 * (dp[a] + dp[o]))).sum(1)
                e = e - 0.5 * (dp * (2.0 * p + dp)).sum(1)
                e = e.index_add(0, a, 0.5 * T).index_add(0, o, -0.5 * T)
            p = p + dp
        if c["project"]:
            e = torch.cat([e[o] - (x - x0) / r[0] for o, r, x, x0 in zip(own, reps, energies(U, p, e), E0)])
    return {"q": q, "p": p, "eps": e}


def exact(case, seed):
    """What run() returns, in 64 bits. None where the sequence of pair maps is long (a Python loop orders
    them) and for the shock tube and the batch of millions of particles."""
    c = case
    reps = _replicas(c)
    n = sum(r[0] for r in reps)
    if c["family"] in ("shock", "batch") or n * max(1, c["steps"]) > 4000000 or (
            c["scheme"] in ("SSA", "HYBRID") and n * c["steps"] * _r_cut(c) ** 3 > 1200000):
        return None
    dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
    return _exact_steps(c, seed, reps, *_state(c, seed, dev))
