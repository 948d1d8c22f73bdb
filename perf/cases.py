"""The work that the speed of this framework is judged by, through its public calls.

What a program does with the library: advance a system by a stretch of time steps and take
its state out ("step"), evaluate a configuration that is new to it ("evaluate"), fit pair
parameters to forces ("match"), run the paper's many-body copper ("copper") and advance an
ensemble of independent systems ("ensemble").  Every call here runs on torch's current
stream with device arrays, as a program that keeps its data on the GPU makes it.
"""
import math

import numpy as np
import torch

from paper_1305_4196_gb300 import autograd as AG
from paper_1305_4196_gb300 import batch as BA
from paper_1305_4196_gb300 import mdgb as M
from paper_1305_4196_gb300 import workloads as W

R_CUT, SKIN, DT = 2.5, 0.3, 0.005
CU_SKIN, CU_DT, CU_KT, CU_A = 0.4, 0.0982, 0.02585, 3.615
# Kob-Andersen 80:20 mixture: the reference parameters and the perturbed ones of a fit
KA_EPS, KA_SIG = ((1.0, 1.5), (1.5, 0.5)), ((1.0, 0.8), (0.8, 0.88))
KA_EPS1, KA_SIG1 = ((1.1, 1.35), (1.35, 0.55)), ((0.9, 0.88), (0.88, 0.792))


def listed():
    return [
        # one configuration of the smallest box the cell grid takes in earnest: a force
        # server called once per configuration (latency, launches, the build of a new state)
        dict(name="evaluate_2k", kind="evaluate", precision="mixed", nx=8, ny=8, nz=8, missing=0, rho=0.8442, T=0.72),
        # the same of a large system: binning, lists, forces, energy and virial of new positions
        dict(name="evaluate_1m", kind="evaluate", precision="mixed", nx=64, ny=64, nz=64, missing=0, rho=0.8442,
             T=0.72),
        # reference forces in double precision for a sample of ordinary size, ragged sides and
        # a few vacancies
        dict(name="evaluate_fp64_360k", kind="evaluate", precision="fp64", nx=41, ny=44, nz=50, missing=97,
             rho=0.8442, T=0.72),
        # the plain method's size, in double precision: a short trajectory of a small liquid
        dict(name="step_fp64_4k", kind="step", precision="fp64", half=False, nx=10, ny=10, nz=10, missing=0,
             rho=0.8442, T=0.72, steps=20),
        # small, ordinary and large liquids in the default precision and list kind: production
        # molecular dynamics between two frames that are written out
        dict(name="step_32k", kind="step", precision="mixed", half=False, nx=20, ny=20, nz=20, missing=0, rho=0.8442,
             T=0.72, steps=20),
        dict(name="step_257k", kind="step", precision="mixed", half=False, nx=37, ny=40, nz=43, missing=5,
             rho=0.8442, T=0.72, steps=20),
        dict(name="step_2m", kind="step", precision="mixed", half=False, nx=80, ny=80, nz=80, missing=0, rho=0.8442,
             T=0.72, steps=20),
        # an inhomogeneous system of about the paper's nanoparticle size: a slab and particles
        # in vacuum, most of the box empty
        dict(name="slab_1m", kind="slab", L=164.0, T=0.3, steps=20),
        # the paper's Newton-3 half lists in colour phases
        dict(name="step_half_108k", kind="step", precision="mixed", half=True, nx=30, ny=30, nz=30, missing=0,
             rho=0.8442, T=0.72, steps=20),
        # one training step of force matching on a snapshot of a binary mixture: forces at the
        # current parameters, loss, gradients to parameters and positions in torch's default type
        dict(name="match_32k", kind="match", precision="mixed", n_cells=20),
        # the paper's bulk copper crystal with its many-body potential
        dict(name="copper_500k", kind="copper", nx=50, ny=50, nz=50, steps=20),
        # replicas of uneven size in one launch, then the forces and energies a sampler reads
        dict(name="ensemble_128", kind="ensemble", systems=128, n_min=256, n_max=32768, steps=10),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _sides(rng, lo, hi):
    """Three unequal cell counts whose product spans lo^3 .. hi^3 over its logarithm."""
    m = _log(rng, lo, hi)
    return [min(hi, max(lo, int(round(m * rng.uniform(0.9, 1.1))))) for _ in range(3)]


def draw(rng):
    kind = rng.choice(["evaluate", "evaluate", "step", "step", "step", "slab", "match", "copper", "ensemble"])
    if kind == "evaluate":
        fp64 = rng.random() < 0.3
        nx, ny, nz = _sides(rng, 8, 44 if fp64 else 64)
        return dict(kind=kind, precision="fp64" if fp64 else "mixed", nx=nx, ny=ny, nz=nz, missing=rng.randint(0, 99),
                    rho=round(rng.uniform(0.75, 0.9), 4), T=round(rng.uniform(0.5, 1.2), 3))
    if kind == "step":
        how = rng.choice(["mixed", "mixed", "mixed", "fp64", "half"])
        nx, ny, nz = _sides(rng, *{"mixed": (10, 76), "fp64": (10, 24), "half": (15, 36)}[how])
        return dict(kind=kind, precision="fp64" if how == "fp64" else "mixed", half=how == "half", nx=nx, ny=ny, nz=nz,
                    missing=rng.randint(0, 99), rho=round(rng.uniform(0.78, 0.88), 4),
                    T=round(rng.uniform(0.5, 1.0), 3), steps=rng.randint(10, 24))
    if kind == "slab":
        return dict(kind=kind, L=round(rng.uniform(110.0, 164.0), 2), T=0.3, steps=rng.randint(10, 20))
    if kind == "match":
        return dict(kind=kind, precision=rng.choice(["mixed", "fp64"]), n_cells=int(round(_log(rng, 9, 22))))
    if kind == "copper":
        nx, ny, nz = _sides(rng, 10, 48)
        return dict(kind=kind, nx=nx, ny=ny, nz=nz, steps=rng.randint(10, 20))
    return dict(kind=kind, systems=rng.randint(8, 120), n_min=256, n_max=rng.choice([2000, 8192, 32768]),
                steps=rng.randint(5, 10))


# ---------------------------------------------------------------- inputs
def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _lattice(nx, ny, nz, a, missing, jitter, g):
    """fcc sites of nx x ny x nz cells of side a, `missing` of them left empty, every
    coordinate displaced by jitter * N(0, 1) and wrapped into the box."""
    d = dict(device="cuda", dtype=torch.float64)
    z, y, x = torch.meshgrid(torch.arange(nz, **d), torch.arange(ny, **d), torch.arange(nx, **d), indexing="ij")
    cells = torch.stack([x.reshape(-1), y.reshape(-1), z.reshape(-1)], 1)
    basis = torch.tensor([[0.0, 0.0, 0.0], [0.5, 0.5, 0.0], [0.5, 0.0, 0.5], [0.0, 0.5, 0.5]], **d)
    pos = ((cells[:, None, :] + basis) * a).reshape(-1, 3)
    box = torch.tensor([nx * a, ny * a, nz * a], **d)
    if missing:
        keep = torch.randperm(len(pos), generator=g, device="cuda")[missing:]
        pos = pos[torch.sort(keep).values]
    pos = torch.remainder(pos + jitter * torch.randn(pos.shape, generator=g, **d), box)
    return torch.where(pos >= box, torch.zeros_like(pos), pos).contiguous(), box


def _velocities(n, kT, mass, g):
    v = torch.randn((n, 3), generator=g, device="cuda", dtype=torch.float64)
    v = v - v.mean(0)
    return (v * torch.sqrt(kT * (3 * n - 3) / (mass * (v * v).sum()))).contiguous()


def _liquid(c, seed):
    """A dense liquid's disorder: fcc sites at the given density, 0.05 sigma of jitter, thermal
    velocities."""
    g = _gen(seed)
    pos, box = _lattice(c["nx"], c["ny"], c["nz"], (4.0 / c["rho"]) ** (1.0 / 3.0), c["missing"], 0.05, g)
    return pos, _velocities(len(pos), c["T"], 1.0, g), box


def _slab(c, seed):
    """The geometry belongs to the case; displacements and velocities to the seed."""
    w = W.slab_nanoparticles(c["L"], rho=0.8442, T=c["T"], seed=3)
    g = _gen(seed)
    box = torch.as_tensor(w.box, device="cuda")
    pos = torch.as_tensor(w.pos, device="cuda")
    pos = torch.remainder(pos + 0.05 * torch.randn(pos.shape, generator=g, device="cuda", dtype=torch.float64), box)
    pos = torch.where(pos >= box, torch.zeros_like(pos), pos).contiguous()
    return pos, _velocities(len(pos), c["T"], 1.0, g), box


def _copper(c, seed):
    g = _gen(seed)
    pos, box = _lattice(c["nx"], c["ny"], c["nz"], CU_A, 0, 0.08, g)
    return pos, _velocities(len(pos), CU_KT, W.copper_tbsma()["mass"], g), box


def _mixture(c, seed):
    """A snapshot of the mixture in float32 or float64, the type its fit runs in, and target
    forces of the size the reference parameters give."""
    g = _gen(seed)
    dt = torch.float64 if c["precision"] == "fp64" else torch.float32
    n = c["n_cells"]
    pos, box = _lattice(n, n, n, (4.0 / 1.2) ** (1.0 / 3.0), 0, 0.05, g)
    pos = pos.to(dt)
    sp = torch.zeros(len(pos), dtype=torch.int32, device="cuda")
    sp[torch.randperm(len(pos), generator=g, device="cuda")[: len(pos) // 5]] = 1
    target = 30.0 * torch.randn(pos.shape, generator=g, device="cuda", dtype=torch.float64)
    eps, sig = (torch.tensor(t, dtype=dt, requires_grad=True) for t in (KA_EPS1, KA_SIG1))
    return pos.requires_grad_(True), box, sp, target, eps, sig


def _replicas(c, seed):
    """Independent systems: atom counts log-uniform, densities U(0.7, 0.95), temperatures
    U(0.5, 1.5).  The sizes belong to the case, the configurations to the seed."""
    rng = np.random.RandomState(c["systems"] * 7919 + c["n_max"])
    g = _gen(seed)
    parts = []
    for _ in range(c["systems"]):
        n = int(round(math.exp(rng.uniform(math.log(c["n_min"]), math.log(c["n_max"])))))
        side = (n / rng.uniform(0.7, 0.95)) ** (1.0 / 3.0)
        nc = 1
        while 4 * nc ** 3 < n:
            nc += 1
        pos, box = _lattice(nc, nc, nc, side / nc, 4 * nc ** 3 - n, 0.05, g)
        parts.append((pos, _velocities(n, rng.uniform(0.5, 1.5), 1.0, g), box))
    return parts


def _n_atoms(c):
    if c["kind"] == "match":
        return 4 * c["n_cells"] ** 3
    if c["kind"] == "slab":
        return int(0.27 * c["L"] ** 3)
    if c["kind"] == "ensemble":
        rng = np.random.RandomState(c["systems"] * 7919 + c["n_max"])
        n = 0
        for _ in range(c["systems"]):
            n += int(round(math.exp(rng.uniform(math.log(c["n_min"]), math.log(c["n_max"])))))
            rng.uniform(0.7, 0.95), rng.uniform(0.5, 1.5)
        return n
    return 4 * c["nx"] * c["ny"] * c["nz"] - c.get("missing", 0)


# ---------------------------------------------------------------- the calls
def prepare(case, seed):
    """The system a program has created and loaded, and the device buffers it reads into."""
    k = case["kind"]
    stream = torch.cuda.current_stream().cuda_stream or None
    if k == "match":
        pos, box, sp, target, eps, sig = _mixture(case, seed)
        s = M.System(len(pos), box.cpu().numpy(), r_cut=R_CUT, skin=SKIN, eps=np.array(KA_EPS), sigma=np.array(KA_SIG),
                     mass=[1.0, 1.0], dt=DT, precision=M.MD_FP64 if case["precision"] == "fp64" else M.MD_MIXED,
                     rcut=R_CUT * np.array(KA_SIG), stream=stream)
        return dict(kind=k, s=s, pos=pos, sp=sp, target=target, eps=eps, sig=sig, rcut=R_CUT * np.array(KA_SIG))
    if k == "ensemble":
        parts = _replicas(case, seed)
        b = BA.Batch([len(p) for p, _, _ in parts], np.stack([x.cpu().numpy() for _, _, x in parts]), r_cut=R_CUT,
                     skin=SKIN, dt=DT, stream=stream)
        pos, vel = torch.cat([p for p, _, _ in parts]), torch.cat([v for _, v, _ in parts])
        b.set_state(pos, vel)
        return dict(kind=k, b=b, steps=case["steps"], f=torch.empty_like(pos))
    if k == "copper":
        P = W.copper_tbsma()
        pos, vel, box = _copper(case, seed)
        s = M.System(len(pos), box.cpu().numpy(), r_cut=P["rc"], skin=CU_SKIN, mass=P["mass"], dt=CU_DT,
                     precision=M.MD_MIXED, stream=stream)
        s.set_tbsma(P["A"], P["xi"], P["p"], P["q"], P["r0"], P["rc"])
        s.set_state(pos, vel)
    else:
        pos, vel, box = (_slab if k == "slab" else _liquid)(case, seed)
        s = M.System(len(pos), box.cpu().numpy(), r_cut=R_CUT, skin=SKIN, dt=DT,
                     precision=M.MD_FP64 if case.get("precision") == "fp64" else M.MD_MIXED,
                     list_kind=M.MD_LIST_HALF_COLOUR8 if case.get("half") else M.MD_LIST_FULL, stream=stream)
        if k == "evaluate":
            return dict(kind=k, s=s, pos=pos, vel=vel, f=torch.empty_like(pos))
        s.set_state(pos, vel)
    return dict(kind=k, s=s, steps=case["steps"], box=box, pos=torch.empty_like(pos), vel=torch.empty_like(pos),
                img=torch.empty(pos.shape, dtype=torch.int32, device="cuda"))


def run(st):
    k = st["kind"]
    if k == "evaluate":
        st["s"].set_state(st["pos"], st["vel"])
        f = st["s"].forces(out=st["f"])
        pe, ke, virial = st["s"].energy_virial()
        return dict(forces=f, pe=pe, ke=ke, virial=virial)
    if k == "match":
        for t in (st["pos"], st["eps"], st["sig"]):
            t.grad = None
        f = AG.lj_forces(st["pos"], st["eps"], st["sig"], st["s"], st["sp"], st["rcut"])
        loss = ((f - st["target"]) ** 2).mean()
        loss.backward()
        return dict(forces=f, loss=loss, pos=st["pos"].grad, eps=st["eps"].grad, sigma=st["sig"].grad)
    if k == "ensemble":
        st["b"].step(st["steps"])
        f = st["b"].forces(out=st["f"])
        pe, ke = st["b"].energies()
        return dict(forces=f, pe=pe, ke=ke)
    # a stretch of the trajectory, then its frame: unwrapped positions and velocities
    st["s"].step(st["steps"])
    M.md_get_state(st["s"].handle, st["pos"], st["vel"], st["img"])
    return dict(pos=st["pos"] + st["img"] * st["box"], vel=st["vel"])


def work(case):
    """Per force evaluation the pairs inside the cutoff, once each (about 33 operations; the
    many-body potential's two passes about 60, the fit's forward and backward pass about 100);
    per time step positions and velocities read and written (96 B per atom); for one
    evaluation positions and velocities read and forces written (72 B), for the fit also the
    targets, and the gradients written."""
    n, k = _n_atoms(case), case["kind"]
    rho, rc, ops = 0.8442, R_CUT, 33.0
    if k == "copper":
        rho, rc, ops = 4.0 / CU_A ** 3, W.copper_tbsma()["rc"], 60.0
    if k == "match":
        rho, ops = 1.2, 100.0
    pairs = 0.5 * n * 4.0 / 3.0 * math.pi * rc ** 3 * case.get("rho", rho)
    if k == "match":
        return dict(bytes=n * (3 * (8 if case["precision"] == "fp64" else 4) * 2 + 4 + 48), flops=ops * pairs)
    if k == "evaluate":
        return dict(bytes=72 * n, flops=ops * pairs)
    evals = case["steps"] + (2 if k == "ensemble" else 0)
    return dict(bytes=96 * n * case["steps"] + (24 * n if k == "ensemble" else 48 * n), flops=ops * pairs * evals)


# ---------------------------------------------------------------- the same in 64 bits, in plain torch
def _pairs(pos, box, r):
    """Every pair (i, j) once with minimum-image distance below r."""
    n = len(pos)
    nc = [max(1, int(x)) for x in (box / (r * 1.0001)).tolist()]
    if min(nc) < 3 or n < 1500:
        out = []
        for lo in range(0, n, max(1, 20_000_000 // n)):
            hi = min(n, lo + max(1, 20_000_000 // n))
            d = pos[lo:hi, None, :] - pos[None, :, :]
            d = d - box * torch.round(d / box)
            near = ((d * d).sum(-1) < r * r).nonzero()
            near[:, 0] += lo
            out.append(near[near[:, 0] < near[:, 1]])
        p = torch.cat(out)
        return p[:, 0], p[:, 1]
    ncv = torch.tensor(nc, device=pos.device)
    c = torch.minimum((torch.remainder(pos, box) / (box / ncv)).long(), ncv - 1)
    cell = c[:, 0] + nc[0] * (c[:, 1] + nc[1] * c[:, 2])
    count = torch.bincount(cell, minlength=nc[0] * nc[1] * nc[2])
    order = torch.argsort(cell, stable=True)
    start = torch.cumsum(count, 0) - count
    cap = int(count.max())
    table = torch.full((len(count), cap), -1, dtype=torch.long, device=pos.device)
    rank = torch.arange(n, device=pos.device) - start[cell[order]]
    table[cell[order], rank] = order
    full = count.nonzero()[:, 0]
    I, J = [], []
    step = max(1, 30_000_000 // (cap * cap))
    for off in [(x, y, z) for z in (0, 1) for y in (-1, 0, 1) for x in (-1, 0, 1) if (z, y, x) >= (0, 0, 0)]:
        for lo in range(0, len(full), step):
            a = full[lo:lo + step]
            ax, ay, az = a % nc[0], (a // nc[0]) % nc[1], a // (nc[0] * nc[1])
            b = (ax + off[0]) % nc[0] + nc[0] * ((ay + off[1]) % nc[1] + nc[1] * ((az + off[2]) % nc[2]))
            i, j = table[a][:, :, None].expand(-1, -1, cap), table[b][:, None, :].expand(-1, cap, -1)
            ok = (i >= 0) & (j >= 0)
            if off == (0, 0, 0):
                ok &= i < j
            i, j = i[ok], j[ok]
            d = pos[i] - pos[j]
            d -= box * torch.round(d / box)
            near = (d * d).sum(-1) < r * r
            I.append(i[near])
            J.append(j[near])
    return torch.cat(I), torch.cat(J)


def _lj(pos, box, pairs, want=False):
    """Forces of the unshifted Lennard-Jones pair potential (and energy, virial)."""
    i, j = pairs
    d = pos[i] - pos[j]
    d -= box * torch.round(d / box)
    r2 = (d * d).sum(-1)
    inside = r2 < R_CUT * R_CUT
    s6 = (1.0 / r2) ** 3
    fr = torch.where(inside, 24.0 * (2.0 * s6 * s6 - s6) / r2, torch.zeros_like(r2))
    p = fr[:, None] * d
    f = torch.zeros_like(pos).index_add_(0, i, p).index_add_(0, j, -p)
    if not want:
        return f
    pe = float(torch.where(inside, 4.0 * (s6 * s6 - s6), torch.zeros_like(r2)).sum())
    vir = [float((d[:, a] * p[:, b]).sum()) for a, b in ((0, 0), (1, 1), (2, 2), (0, 1), (0, 2), (1, 2))]
    return f, pe, np.array(vir)


def _tbsma(pos, box, pairs, P):
    i, j = pairs
    d = pos[i] - pos[j]
    d -= box * torch.round(d / box)
    r = torch.sqrt((d * d).sum(-1))
    inside = r < P["rc"]
    zero = torch.zeros_like(r)
    x = r / P["r0"] - 1.0
    psi = torch.where(inside, P["xi"] ** 2 * torch.exp(-2.0 * P["q"] * x), zero)
    phi = torch.where(inside, P["A"] * torch.exp(-P["p"] * x), zero)
    rho = torch.zeros(len(pos), dtype=pos.dtype, device=pos.device).index_add_(0, i, psi).index_add_(0, j, psi)
    inv = 1.0 / torch.sqrt(rho)
    p = ((2.0 * P["p"] / P["r0"] * phi - P["q"] / P["r0"] * psi * (inv[i] + inv[j])) / r)[:, None] * d
    return torch.zeros_like(pos).index_add_(0, i, p).index_add_(0, j, -p)


def _verlet(pos, vel, box, steps, dt, mass, force, reach):
    """Velocity Verlet from (pos, vel); force(pos, pairs) over pairs closer than `reach` plus a
    margin, found anew when an atom has moved half of it."""
    margin = 0.6
    pos, vel, ref, pairs = pos.clone(), vel.clone(), None, None
    for step in range(steps + 1):
        if ref is None or float((pos - ref).square().sum(1).max()) > (0.5 * margin) ** 2:
            ref, pairs = pos.clone(), _pairs(pos, box, reach + margin)
        f = force(pos, pairs)
        if step > 0:
            vel += 0.5 * dt / mass * f
        if step == steps:
            break
        vel += 0.5 * dt / mass * f
        pos += dt * vel
    return pos, vel


def exact(case, seed):
    k = case["kind"]
    if k == "evaluate":
        pos, vel, box = _liquid(case, seed)
        f, pe, vir = _lj(pos, box, _pairs(pos, box, R_CUT), want=True)
        return dict(forces=f, pe=pe, ke=float(0.5 * (vel * vel).sum()), virial=vir)
    if k == "match":
        pos, box, sp, target, eps, sig = _mixture(case, seed)
        p, e, s = (t.detach().to("cuda", torch.float64).requires_grad_(True) for t in (pos, eps, sig))
        rc = R_CUT * torch.tensor(KA_SIG, device="cuda", dtype=torch.float64)
        i, j = _pairs(p.detach(), box, R_CUT)
        d = p[i] - p[j]
        d = d - box * torch.round(d.detach() / box)
        a, b = sp[i].long(), sp[j].long()
        r2 = (d * d).sum(-1)
        keep = (r2.detach() < rc[a, b] ** 2).nonzero()[:, 0]
        i, j, d, a, b, r2 = i[keep], j[keep], d[keep], a[keep], b[keep], r2[keep]
        s6 = (s[a, b] ** 2 / r2) ** 3
        q = (24.0 * e[a, b] * (2.0 * s6 * s6 - s6) / r2)[:, None] * d
        f = torch.zeros_like(p).index_add(0, i, q).index_add(0, j, -q)
        loss = ((f - target) ** 2).mean()
        loss.backward()

        def shared(t):  # entries [a][b] and [b][a] are one value
            return t + t.T - torch.diag(torch.diagonal(t))

        return dict(forces=f.detach(), loss=loss.detach(), pos=p.grad, eps=shared(e.grad), sigma=shared(s.grad))
    if k == "ensemble":
        F, PE, KE = [], [], []
        for pos, vel, box in _replicas(case, seed):
            pos, vel = _verlet(pos, vel, box, case["steps"], DT, 1.0, lambda x, pr: _lj(x, box, pr), R_CUT)
            f, pe, _ = _lj(pos, box, _pairs(pos, box, R_CUT), want=True)
            F.append(f)
            PE.append(pe)
            KE.append(float(0.5 * (vel * vel).sum()))
        return dict(forces=torch.cat(F), pe=np.array(PE), ke=np.array(KE))
    if k == "copper":
        P = W.copper_tbsma()
        pos, vel, box = _copper(case, seed)
        pos, vel = _verlet(pos, vel, box, case["steps"], CU_DT, P["mass"], lambda x, pr: _tbsma(x, box, pr, P), P["rc"])
        return dict(pos=pos, vel=vel)
    pos, vel, box = (_slab if k == "slab" else _liquid)(case, seed)
    pos, vel = _verlet(pos, vel, box, case["steps"], DT, 1.0, lambda x, pr: _lj(x, box, pr), R_CUT)
    return dict(pos=pos, vel=vel)
