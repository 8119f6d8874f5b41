"""What is timed: the work a user of this library has it do, through its public
entry points (``mtpt.Simulation`` / ``Batch`` and the ``mtpt_*`` calls,
``autograd.mtpt_run``).

A case is a dict of plain values; ``kind`` says which entry points it goes
through:

* ``run``      a handle that keeps its particles: a number of time steps, then
               the masses and positions read into device tensors;
* ``noalloc``  one step on the caller's own device buffers;
* ``batch``    an ensemble of independent realisations in one handle;
* ``react``    as ``run`` with the reaction A + B -> 0 (species B is read into
               host memory, as its call does);
* ``stream``   a host loop: load from pinned memory, step, read back, the copies
               overlapped;
* ``grad``     the differentiable run: steps, a binned misfit, its gradient with
               respect to the initial masses and D.

Particles are uniform in a box whose side gives the density ``rho``, as in the
workloads of ``paper_2204_03756_gb300/workloads.py``.
"""
import math

import numpy as np
import torch

from paper_2204_03756_gb300 import autograd, mtpt

FORMS = {"fp64": mtpt.MTPT_FP64, "fp32w": mtpt.MTPT_FP32W}
BINS = 100          # bins per axis of the gradient case's misfit
REACT_K = 1.0       # rate constant of A + B -> 0


def _case(name, kind, dim, n, form, steps, mass, rho=1.0, D=1.0, kappa=0.5, dt=0.1, drift=0.0,
          members=1, n_min=0):
    return {"name": name, "kind": kind, "dim": dim, "n": n, "form": form, "steps": steps,
            "mass": mass, "rho": rho, "D": D, "kappa": kappa, "dt": dt, "drift": drift,
            "members": members, "n_min": n_min}


def listed():
    return [
        # a loop that looks at the state after every step of the small validation problem
        _case("one step 2d fp64", "run", 2, 10_000, "fp64", 1, "half"),
        # the small validation problem, run whole
        _case("100 steps 2d fp64", "run", 2, 10_000, "fp64", 100, "half"),
        # a step inside a program that owns all device memory
        _case("noalloc 2d fp32w", "noalloc", 2, 20_011, "fp32w", 1, "half"),
        # the large 2-d run, in both forms
        _case("large 2d fp32w", "run", 2, 4_000_000, "fp32w", 20, "spot"),
        _case("large 2d fp64", "run", 2, 4_000_000, "fp64", 5, "spot"),
        # the large 3-d run
        _case("large 3d fp32w", "run", 3, 2_000_000, "fp32w", 20, "half", dt=0.05),
        # an ordinary 3-d run at an odd size, with a uniform velocity
        _case("odd 3d fp64 drift", "run", 3, 250_007, "fp64", 8, "uniform", dt=0.05, drift=0.01),
        # the paper's own 2-d problem: 1e7 particles at density 10 (about 57 neighbours each)
        _case("dense 2d fp32w", "run", 2, 10_000_000, "fp32w", 4, "half", rho=10.0),
        # the ensemble: realisations of 5e3 to 2e5 particles, each with its own D and density
        _case("ensemble 2d fp32w", "batch", 2, 200_000, "fp32w", 5, "half", members=512,
              n_min=5_000),
        # a fast reaction front between two species
        _case("reaction 2d fp32w", "react", 2, 1_000_003, "fp32w", 20, "half"),
        # one step per state that arrives from, and goes back to, host memory
        _case("host stream 2d fp32w", "stream", 2, 4_000_000, "fp32w", 1, "spot"),
        # gradient of a misfit through the whole run, a checkpoint every 20 steps
        _case("gradient 2d", "grad", 2, 250_000, "fp32w", 200, "uniform", D=0.5),
    ]


def _neighbours(c):
    """Expected neighbours of a particle: density x volume of the cutoff ball."""
    psi = math.sqrt(36.0 * (1.0 - c["kappa"]) * c["D"] * c["dt"])
    return c["rho"] * {1: 2.0 * psi, 2: math.pi * psi ** 2, 3: 4.0 / 3.0 * math.pi * psi ** 3}[c["dim"]]


def _cost(c):
    total = c["members"] * c["n"] if c["kind"] == "batch" else c["n"]
    factor = {"grad": 8.0, "stream": 4.0, "batch": 0.4}.get(c["kind"], 1.0)
    return factor * total * c["steps"] * (10.0 + _neighbours(c)) * (2.0 if c["form"] == "fp64" else 1.0)


def draw(rng):
    def spread(lo, hi):
        return math.exp(rng.uniform(math.log(lo), math.log(hi)))

    limit = _cost(listed()[7])
    kind = rng.choice(["run"] * 6 + ["noalloc", "batch", "react", "stream", "grad"])
    dim = 2 if kind in ("batch", "grad") else rng.choice([2, 2, 2, 3, 3, 1])
    top = {"noalloc": 65_536, "batch": 200_000, "react": 2_000_000, "stream": 4_000_000,
           "grad": 250_000, "run": 4_000_000}[kind]
    c = _case("", kind, dim, int(spread(1_000, top)) | 1, rng.choice(["fp64", "fp32w"]),
              rng.choice([1, 2, 5, 10, 20, 50, 100]), rng.choice(["half", "spot", "uniform"]),
              rho=round(spread(0.5, 4.0 if dim == 3 else 10.0), 3), D=round(rng.uniform(0.1, 2.0), 3),
              kappa=rng.choice([0.25, 0.5, 0.75]), dt=0.05 if dim == 3 else 0.1,
              drift=rng.choice([0.0, 0.0, 0.0, 0.01]))
    del c["name"]
    if kind == "batch":
        c.update(members=int(spread(8, 512)), n_min=1 + c["n"] // 40)
    if kind in ("noalloc", "stream"):
        c["steps"] = 1
    if kind == "grad":
        c.update(mass="uniform", drift=0.0)
    while c["steps"] > 1 and _cost(c) > limit:
        c["steps"] = max(1, c["steps"] // 2)
    while _cost(c) > limit:
        c["n"] = (c["n"] // 2) | 1
    return c


# --- inputs -------------------------------------------------------------------

def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _counts(c):
    """Particle counts of a batch's realisations, log-uniform: the case's, whatever the seed."""
    rng = np.random.default_rng(c["members"])
    return np.exp(rng.uniform(math.log(c["n_min"]), math.log(c["n"]), c["members"])).astype(np.int64)


def _members(c, seed):
    """(n, box side, D, walk seed) of every realisation."""
    if c["kind"] != "batch":
        return [(c["n"], (c["n"] / c["rho"]) ** (1.0 / c["dim"]), c["D"], seed)]
    k = c["members"]
    n = _counts(c)
    rng = np.random.default_rng(seed)
    rho, D = c["rho"] * rng.uniform(0.5, 2.0, k), c["D"] * rng.uniform(0.1, 2.0, k)
    return [(int(n[i]), math.sqrt(n[i] / rho[i]), float(D[i]), seed + 1 + i) for i in range(k)]


def _params(c, member):
    n, side, D, seed = member
    d = c["dim"]
    return mtpt.Params(dim=d, D=D, kappa=c["kappa"], dt=c["dt"], lo=(0.0,) * d, hi=(side,) * d,
                       seed=seed, precision=FORMS[c["form"]],
                       v=(c["drift"], 0.5 * c["drift"], 0.0) if c["drift"] else (0.0, 0.0, 0.0))


def _particles(c, seed, members):
    """Positions (dim x n) and masses (n) on the GPU, members one after another."""
    g = _generator(seed)
    counts = torch.tensor([m[0] for m in members], device="cuda")
    side = torch.tensor([m[1] for m in members], dtype=torch.float64, device="cuda")
    side = torch.repeat_interleave(side, counts)
    pos = torch.rand((c["dim"], side.numel()), generator=g, dtype=torch.float64, device="cuda") * side
    if c["mass"] == "half":
        mass = (pos[0] < 0.5 * side).double()
    elif c["mass"] == "spot":
        mass = torch.exp(-((pos - 0.5 * side) ** 2).sum(0) / 50.0)
    else:
        mass = torch.rand(side.numel(), generator=g, dtype=torch.float64, device="cuda")
    return pos, mass


def _target(c, side, seed):
    phase = np.random.default_rng(seed).uniform(0.0, 1.0, 2)
    x = (torch.arange(BINS, device="cuda", dtype=torch.float64) + 0.5) / BINS * (2.0 * math.pi)
    return c["rho"] * (0.5 + 0.25 * torch.outer(torch.sin(x + 2.0 * math.pi * phase[0]),
                                                torch.cos(x + 2.0 * math.pi * phase[1])))


def prepare(case, seed):
    c, members = case, _members(case, seed)
    pos, mass = _particles(c, seed, members)
    n, d = mass.numel(), c["dim"]
    s = {"case": c, "mass": torch.empty_like(mass), "pos": torch.empty_like(pos)}
    if c["kind"] == "batch":
        s["sim"] = mtpt.Batch([_params(c, m) for m in members], [m[0] for m in members],
                              pos.cpu().numpy(), mass.cpu().numpy())
        return s
    s["params"] = p = _params(c, members[0])
    if c["kind"] == "noalloc":
        s.update(pos=pos, mass=mass, step=0)
        return s
    if c["kind"] == "grad":
        s.update(pos=pos, mass=mass.requires_grad_(),
                 D=torch.tensor(c["D"], dtype=torch.float64, requires_grad=True),
                 target=_target(c, members[0][1], seed))
        return s
    s["sim"] = sim = mtpt.Simulation(p)
    if c["kind"] == "stream":
        s.update(host_pos=pos.cpu().pin_memory(), host_mass=mass.cpu().pin_memory(),
                 out=torch.empty(n, dtype=torch.float64).pin_memory())
        sim.set_particles(s["host_pos"].numpy(), s["host_mass"].numpy())
        return s
    mtpt.mtpt_set_particles_device(sim.h, d, pos, mass)
    sim.n = n
    if c["kind"] == "react":
        sim.set_reaction(REACT_K, (1.0 - mass).clamp_(min=0.0).cpu().numpy())
    return s


def run(state):
    s, c = state, state["case"]
    if c["kind"] == "noalloc":
        mtpt.mtpt_step_noalloc(s["params"], s["step"], s["pos"], s["mass"])
        s["step"] += 1
        return {"mass": s["mass"], "pos": s["pos"]}
    if c["kind"] == "grad":
        p = s["params"]
        mass, pos = autograd.mtpt_run(s["mass"], s["D"], p, s["pos"], c["steps"], 20)
        conc = autograd.binned_concentration(pos, mass, p.lo, p.hi, (BINS, BINS))
        loss = ((conc - s["target"]) ** 2).sum()
        g_mass, g_D = torch.autograd.grad(loss, (s["mass"], s["D"]))
        return {"mass": mass.detach(), "pos": pos, "conc": conc.detach(), "g_mass": g_mass, "g_D": g_D}
    sim = s["sim"]
    if c["kind"] == "stream":
        sim.set_particles_async(s["host_pos"], s["host_mass"])
        sim.step(c["steps"])
        sim.masses_async(s["out"])
        return {"mass": s["out"]}
    sim.step(c["steps"])
    mtpt.mtpt_get_masses_device(sim.h, s["mass"])
    mtpt.mtpt_get_positions_device(sim.h, s["pos"])
    out = {"mass": s["mass"], "pos": s["pos"]}
    if c["kind"] == "react":
        out["mass_b"] = sim.masses_b()
    return out


def work(case):
    """Per step: every particle's state read and written once; per ordered pair the
    distance, kernel, weight and flux; per particle the walk's draws."""
    c = case
    n = int(_counts(c).sum()) if c["kind"] == "batch" else c["n"]
    d, species = c["dim"], 2 if c["kind"] == "react" else 1
    nb = _neighbours(c)
    sweeps = 3 if c["kind"] == "grad" else 1    # forward, recomputation, adjoint
    return {"bytes": sweeps * c["steps"] * n * 16.0 * (d + species),
            "flops": sweeps * c["steps"] * n * (nb * (3.0 * d + 9.0 * species) + 60.0)}


def tolerance(case):
    """Positions are one binary64 sum per axis and step.  Masses in the binary64
    form: 6e-17 (one step) to 2e-16 (100 steps) of the largest mass against
    serial sums in another order, and a spot's rms is 1/200 of its largest; the
    gradient's sums over all steps cancel to some 1e-3 of their terms.  In the
    precision form, binary32 weights: 2e-8 of the masses' norm after 20 steps."""
    if case["form"] == "fp64":
        return {"rel": 1e-11, "max": 1e-9} if case["kind"] == "grad" else {"rel": 1e-14, "max": 1e-12}
    return {"rel": 2e-7, "max": 1e-5}


# --- the same in 64 bits --------------------------------------------------------

def _philox(ids, step, seed):
    """Philox4x32-10 words of counters (id, step low, step high, 0) under the seed's key."""
    m32 = 0xFFFFFFFF
    x = [ids.clone(), torch.full_like(ids, step & m32), torch.full_like(ids, step >> 32),
         torch.zeros_like(ids)]
    k0, k1 = seed & m32, (seed >> 32) & m32
    for _ in range(10):
        # 32 x 32 -> 64-bit products: int64 wraps, which leaves both halves right
        p0, p1 = x[0] * 0xD2511F53, x[2] * 0xCD9E8D57
        x = [((p1 >> 32) & m32) ^ x[1] ^ k0, p1 & m32, ((p0 >> 32) & m32) ^ x[3] ^ k1, p0 & m32]
        k0, k1 = (k0 + 0x9E3779B9) & m32, (k1 + 0xBB67AE85) & m32
    return x


def _normals(ids, step, seed, d):
    w = [((v >> 8) + 1).double() / 2.0 ** 24 for v in _philox(ids, step, seed)]
    z = []
    for a in (0, 2):
        r = torch.sqrt(-2.0 * torch.log(w[a]))
        z += [r * torch.cos(2.0 * math.pi * w[a + 1]), r * torch.sin(2.0 * math.pi * w[a + 1])]
    return torch.stack(z[:d])


def _pairs(pos, side, psi):
    """Chunks (i, j) of ordered pairs within psi, indices into the given order."""
    d, n = pos.shape
    ncell = max(1, min(int(side / (psi * (1.0 + 1e-9))), int((4.0 * n + 64.0) ** (1.0 / d))))
    cell = (pos * (ncell / side)).long().clamp_(0, ncell - 1)
    lin = sum(cell[a] * ncell ** a for a in range(d))
    order = torch.argsort(lin)
    count = torch.bincount(lin, minlength=ncell ** d)
    start = torch.cat([count.new_zeros(1), count.cumsum(0)])
    ps, cs = pos[:, order], cell[:, order]
    rows = [(dy, dz) for dy in ((-1, 0, 1) if d > 1 else (0,)) for dz in ((-1, 0, 1) if d > 2 else (0,))]
    mean = max(1.0, 3.0 * n / ncell ** d)
    chunk = max(1024, int(6e7 / mean))
    for b in range(0, n, chunk):
        e = min(n, b + chunk)
        me = torch.arange(b, e, device=pos.device)
        for dy, dz in rows:
            cy, cz = (cs[1, b:e] + dy if d > 1 else None), (cs[2, b:e] + dz if d > 2 else None)
            base, ok = 0, torch.ones(e - b, dtype=torch.bool, device=pos.device)
            for a, ca in ((1, cy), (2, cz)):
                if ca is not None:
                    ok &= (ca >= 0) & (ca < ncell)
                    base = base + ca.clamp(0, ncell - 1) * ncell ** a
            lo = start[base + (cs[0, b:e] - 1).clamp(min=0)]
            hi = start[base + (cs[0, b:e] + 1).clamp(max=ncell - 1) + 1]
            cnt = (hi - lo) * ok
            i = torch.repeat_interleave(me, cnt)
            first = cnt.cumsum(0) - cnt
            j = torch.arange(i.numel(), device=pos.device) + torch.repeat_interleave(lo - first, cnt)
            diff = ps[:, i] - ps[:, j]
            keep = ((diff * diff).sum(0) <= psi * psi) & (i != j)
            yield order[i[keep]], order[j[keep]]


def _transfer(pos, masses, side, psi, h2):
    """One mass-transfer update of every species on fixed positions."""
    few = []
    r = torch.ones_like(masses[0])
    for i, j in _pairs(pos.detach(), side, psi):
        K = torch.exp(-((pos[:, i] - pos[:, j]) ** 2).sum(0) / (2.0 * h2))
        r = r.index_add(0, i, K)
        if few is not None:
            few.append((i, j, K))
            if sum(f[0].numel() for f in few) > 2e8:
                few = None
    out = [m.clone() for m in masses]
    for p in few if few is not None else _pairs(pos, side, psi):
        i, j = p[:2]
        K = p[2] if few is not None else torch.exp(-((pos[:, i] - pos[:, j]) ** 2).sum(0) / (2.0 * h2))
        W = 2.0 * K / (r[i] + r[j])
        out = [o.index_add(0, i, W * (m[j] - m[i])) for o, m in zip(out, masses)]
    return out


def _react(a, b, kp, dt):
    big, small = torch.maximum(a, b), torch.minimum(a, b)
    x = kp * (big - small) * dt
    phi = torch.where(x > 0.0, -torch.expm1(-x) / torch.where(x > 0.0, x, torch.ones_like(x)),
                      torch.ones_like(x))
    q = 1.0 + kp * small * dt * phi
    nb, ns = big / q, small * torch.exp(-x) / q
    nb, ns = torch.where(small < 0.0, big, nb), torch.where(small < 0.0, small, ns)
    return torch.where(a >= b, nb, ns), torch.where(a >= b, ns, nb)


def _member_exact(c, member, pos, masses, D):
    n, side, _, seed = member
    d = c["dim"]
    ids = torch.arange(n, device=pos.device)
    d_mt = (1.0 - c["kappa"]) * D
    sigma = (2.0 * c["kappa"] * D * c["dt"]) ** 0.5
    h2 = 2.0 * d_mt * c["dt"]
    psi = math.sqrt(36.0 * float(d_mt) * c["dt"])
    move = torch.tensor([c["drift"], 0.5 * c["drift"], 0.0][:d], dtype=torch.float64,
                        device=pos.device)[:, None] * c["dt"]
    for t in range(c["steps"]):
        pos = pos + (move + sigma * _normals(ids, t, seed, d))
        for _ in range(4):      # mirrors (a step is far shorter than the box)
            pos = torch.where(pos < 0.0, -pos, pos)
            pos = torch.where(pos > side, 2.0 * side - pos, pos)
        masses = _transfer(pos, masses, side, psi, h2)
        if len(masses) == 2:
            masses = _react(masses[0], masses[1], REACT_K * n / side ** d, c["dt"])
    return pos, masses


def exact(case, seed):
    c, members = case, _members(case, seed)
    pos, mass = _particles(c, seed, members)
    if c["kind"] == "grad":
        mass.requires_grad_()
        D = torch.tensor(c["D"], dtype=torch.float64, device="cuda", requires_grad=True)
        out, (end,) = _member_exact(c, members[0], pos, [mass], D)
        side = members[0][1]
        cell = (out.detach() * (BINS / side)).long().clamp_(0, BINS - 1)
        conc = end.new_zeros(BINS * BINS).index_add(0, cell[0] * BINS + cell[1], end) * (BINS / side) ** 2
        conc = conc.view(BINS, BINS)
        g_mass, g_D = torch.autograd.grad(((conc - _target(c, side, seed)) ** 2).sum(), (mass, D))
        return {"mass": end.detach(), "pos": out.detach(), "conc": conc.detach(), "g_mass": g_mass,
                "g_D": g_D}
    if c["kind"] == "batch":
        ends, first = [], 0
        for m in members:
            part = slice(first, first + m[0])
            ends.append(_member_exact(c, m, pos[:, part], [mass[part]], m[2]))
            first += m[0]
        return {"mass": torch.cat([e[1][0] for e in ends]), "pos": torch.cat([e[0] for e in ends], 1)}
    species = [mass] if c["kind"] != "react" else [mass, (1.0 - mass).clamp(min=0.0)]
    end, masses = _member_exact(c, members[0], pos, species, c["D"])
    if c["kind"] == "stream":
        return {"mass": masses[0].cpu()}
    out = {"mass": masses[0], "pos": end}
    if c["kind"] == "react":
        out["mass_b"] = masses[1].cpu().numpy()
    return out
