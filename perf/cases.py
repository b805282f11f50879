"""The calls this library is timed on, through its public entry points.

A case is a dict of plain values: the kind of call ("step": rebuild and
evaluate; "noalloc": the allocation-free entry point; "fit": one training step
of the force field; "md": molecular-dynamics steps), the system ("lj": a
Lennard-Jones fluid, "water": TIP3P-shaped waters, "chain": a chain molecule
in water) with its size, and the option in use ("none", "pme", "tables",
"host": page-locked host arrays).  "boxes" > 1 is a batch of water boxes of
uneven sizes.  Sizes follow the configurations of bench.py and of the tests.
"""

from __future__ import annotations

import math
from types import SimpleNamespace

import numpy as np
import torch

from paper_0902_0827_gb300 import nb

KE, S14_LJ, S14_C = 332.0636, 0.5, 1.0 / 1.2
Q_O, Q_H, R_OH, THETA = -0.834, 0.417, 0.9572, math.radians(104.52)
R_HH = 2.0 * R_OH * math.sin(0.5 * THETA)
SIG_O, EPS_O = 3.1507, 0.1521
SIG_H, EPS_H = 0.4, 0.046          # CHARMM's TIP3P hydrogen, for fitting and dynamics
WATERS_PER_A3 = 6.02214076e23 / 18.015 * 1e-24
CHAIN_ATOMS_PER_A3 = 23500 / 62.2 ** 3
TABLE_N = 4096
MD = dict(dt=0.001, gamma=5.0, temperature=300.0, seed=2009)
MD_STEPS = 10
FIT_RATE = 1e-6                    # A and kcal/mol per parameter and training step


def listed():
    return [
        # the smallest calls: a plain LJ fluid, and a host application without device allocation
        {"name": "lj_256", "kind": "step", "system": "lj", "atoms": 256, "option": "none"},
        {"name": "noalloc_water_900", "kind": "noalloc", "system": "water", "waters": 300, "option": "none"},
        # a small water box
        {"name": "water_6144", "kind": "step", "system": "water", "waters": 2048, "option": "none"},
        # the solvated-protein size of the headline benchmark: device arrays, page-locked host arrays
        # (a host program's own positions), and the full electrostatics with smooth PME on a 64^3 grid
        {"name": "chain_23500", "kind": "step", "system": "chain", "chain": 2500, "waters": 7000, "option": "none"},
        {"name": "chain_23500_host", "kind": "step", "system": "chain", "chain": 2500, "waters": 7000,
         "option": "host"},
        {"name": "chain_23500_pme", "kind": "step", "system": "chain", "chain": 2500, "waters": 7000,
         "option": "pme"},
        # the tabulated radial functions, on an odd size
        {"name": "water_20001_tables", "kind": "step", "system": "water", "waters": 6667, "option": "tables"},
        # one training step of a force field on one system, and on uneven boxes at once: forces, energies,
        # their adjoint, the parameters updated
        {"name": "chain_23500_fit", "kind": "fit", "system": "chain", "chain": 2500, "waters": 7000,
         "option": "none"},
        {"name": "boxes_16_fit", "kind": "fit", "system": "water", "boxes": 16, "lo": 500, "hi": 20000,
         "option": "none"},
        # dynamics of the solvated chain with PME, ten steps a call
        {"name": "chain_23500_md", "kind": "md", "system": "chain", "chain": 2500, "waters": 7000, "option": "pme"},
        # many replicas in one launch; the largest single system
        {"name": "boxes_64", "kind": "step", "system": "water", "boxes": 64, "lo": 500, "hi": 20000,
         "option": "none"},
        {"name": "water_999999", "kind": "step", "system": "water", "waters": 333333, "option": "none"},
    ]


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    def chain():
        atoms = log_int(3000, 60000)
        n = max(60, int(atoms * rng.uniform(0.05, 0.15)))
        return {"system": "chain", "chain": n, "waters": (atoms - n) // 3}

    kind = rng.choice(["lj", "water", "water", "chain", "host", "pme", "tables", "fit", "boxes_fit", "md", "boxes",
                       "noalloc"])
    if kind == "lj":
        return {"kind": "step", "system": "lj", "atoms": log_int(240, 100000), "option": "none"}
    if kind == "noalloc":
        return {"kind": "noalloc", "system": "water", "waters": log_int(200, 1333), "option": "none"}
    if kind == "water":
        return {"kind": "step", "system": "water", "waters": log_int(199, 250000), "option": "none"}
    if kind == "chain":
        return {"kind": "step", **chain(), "option": "none"}
    if kind == "host":
        return {"kind": "step", **chain(), "option": "host"}
    if kind == "pme":
        return {"kind": "step", **chain(), "option": "pme"}
    if kind == "tables":
        return {"kind": "step", "system": "water", "waters": log_int(199, 30000), "option": "tables"}
    if kind == "fit":
        return {"kind": "fit", **chain(), "option": "none"}
    if kind == "md":
        return {"kind": "md", **chain(), "option": "pme"}
    boxes = rng.randint(2, 12) if kind == "boxes_fit" else rng.randint(2, 64)
    lo = log_int(500, 4000)
    return {"kind": "fit" if kind == "boxes_fit" else "step", "system": "water", "boxes": boxes, "lo": lo,
            "hi": log_int(lo + 500, 20000), "option": "none"}


# ------------------------------------------------------------------- inputs


def _rng(case, seed):
    return np.random.Generator(np.random.PCG64([902827, int(seed)]))


def _rotations(rng, n, dev):
    q = torch.from_numpy(rng.normal(size=(n, 4))).to(dev)
    w, x, y, z = (q / q.norm(dim=1, keepdim=True)).unbind(1)
    return torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y - z * w), 2 * (x * z + y * w),
                        2 * (x * y + z * w), 1 - 2 * (x * x + z * z), 2 * (y * z - x * w),
                        2 * (x * z - y * w), 2 * (y * z + x * w), 1 - 2 * (x * x + y * y)], 1).reshape(n, 3, 3)


def _waters(rng, n, L, dev, avoid=None, clear=1.4):
    """[n, 3, 3] positions (O, H, H) of n waters on a jittered grid with random orientations, redrawn while
    an atom comes within `clear` of another molecule (neighbouring sites and, when given, `avoid`)."""
    side = math.ceil(n ** (1.0 / 3.0))
    while True:
        g = torch.arange(side, device=dev)
        site = torch.stack(torch.meshgrid(g, g, g, indexing="ij"), -1).reshape(-1, 3)
        o = (site + 0.5) * (L / side) + torch.from_numpy(rng.uniform(-0.15, 0.15, (side ** 3, 3))).to(dev)
        ok = torch.arange(side ** 3, device=dev)
        if avoid is not None:
            far = torch.cat([(_image(a[:, None] - avoid[None], L).square().sum(-1).min(1).values > 2.6 ** 2)
                             for a in o.split(4096)])
            ok = ok[far]
        if len(ok) >= n:
            break
        side += 1
    pick = ok[torch.from_numpy(rng.permutation(len(ok))[:n]).to(dev)].sort().values
    o, site = o[pick], site[pick]
    body = torch.tensor([[0.0, 0.0, 0.0], [R_OH * math.cos(THETA / 2), R_OH * math.sin(THETA / 2), 0.0],
                         [R_OH * math.cos(THETA / 2), -R_OH * math.sin(THETA / 2), 0.0]], dtype=torch.float64,
                        device=dev)
    at = torch.full((side ** 3,), -1, dtype=torch.int64, device=dev)
    at[pick] = torch.arange(n, device=dev)
    off = [(i, j, k) for i in (-1, 0, 1) for j in (-1, 0, 1) for k in (-1, 0, 1) if (i, j, k) > (0, 0, 0)]
    R = _rotations(rng, n, dev)
    for _ in range(60):
        x = o[:, None] + torch.einsum("nij,kj->nki", R, body)
        bad = torch.zeros(n, dtype=torch.bool, device=dev)
        for d in off:
            s = (site + torch.tensor(d, device=dev)) % side
            j = at[(s[:, 0] * side + s[:, 1]) * side + s[:, 2]]
            i = torch.nonzero(j >= 0)[:, 0]
            j = j[i]
            hit = _image(x[i][:, :, None] - x[j][:, None], L).square().sum(-1).amin((1, 2)) < clear ** 2
            bad[i[hit]] = True
            bad[j[hit]] = True
        if avoid is not None:
            near = torch.cat([(_image(a[:, :, None] - avoid[None, None], L).square().sum(-1).amin((1, 2))
                               < clear ** 2) for a in x.split(2048)])
            bad |= near
        m = torch.nonzero(bad)[:, 0]
        if len(m) == 0:
            break
        R[m] = _rotations(rng, len(m), dev)
    return x


def _chain(rng, n, L):
    """[n, 3] beads of a self-avoiding walk on a diamond lattice (bonds 1.5 A, tetrahedral angles) inside
    the box, slightly perturbed."""
    steps = [(1, 1, 1), (1, -1, -1), (-1, 1, -1), (-1, -1, 1)]
    unit, half = 1.5 / math.sqrt(3.0), 0.5 * (L - 4.0)
    draws = iter(())
    path, used = [(0, 0, 0)], {(0, 0, 0)}
    while len(path) < n:
        p, s = path[-1], 1 if len(path) % 2 else -1
        done = False
        for _ in range(8):
            k = next(draws, None)
            if k is None:
                draws = iter(rng.integers(0, 4, 4096).tolist())
                k = next(draws)
            c = tuple(a + s * b for a, b in zip(p, steps[k]))
            if c in used or any(abs(a) * unit > half for a in c):
                continue
            if any(t != p and t in used for t in (tuple(a - s * b for a, b in zip(c, v)) for v in steps)):
                continue
            path.append(c)
            used.add(c)
            done = True
            break
        if not done:  # stuck: take back a few beads
            for _ in range(min(len(path) - 1, 12)):
                used.discard(path.pop())
    return np.array(path) * unit + 0.5 * L + rng.normal(0.0, 0.03, (n, 3))


def _image(d, L):
    return d - L * torch.round(d / L)


def _wrapped(x, L):
    """FP32 positions in [0, L)."""
    L32 = torch.tensor(L, dtype=torch.float32, device=x.device)
    p = torch.remainder(x, L32.double()).float()
    return torch.where(p >= L32, torch.zeros_like(p), p).cpu().numpy()


def _system(pos, q, typ, sigma, eps, L, excl, p14=None, cutoff=9.0, alpha=0.32):
    return SimpleNamespace(
        pos=pos, q=np.asarray(q, np.float32), type=np.asarray(typ, np.int32), sigma=np.asarray(sigma, np.float32),
        epsilon=np.asarray(eps, np.float32), box=np.full(3, L, np.float32), excl=np.asarray(excl, np.int32),
        pairs14=np.zeros((0, 2), np.int32) if p14 is None else np.asarray(p14, np.int32), cutoff=cutoff,
        switch_dist=7.5, ewald_alpha=alpha, coulomb_k=KE, scale14_lj=S14_LJ, scale14_coul=S14_C,
        n_atoms=len(pos))


def _water_excl(n, first=0):
    b = first + 3 * np.arange(n)
    return np.concatenate([np.stack([b, b + 1], 1), np.stack([b, b + 2], 1), np.stack([b + 1, b + 2], 1)])


def _box_sizes(case):
    """Waters of each box of a batch: atom counts log-uniform in [lo, hi], the same for every seed."""
    rng = np.random.Generator(np.random.PCG64([case["boxes"], case["lo"], case["hi"]]))
    atoms = np.exp(rng.uniform(math.log(case["lo"]), math.log(case["hi"]), case["boxes"]))
    return [max(199, int(round(a / 3))) for a in atoms]


def _systems(case, seed):
    """The case's systems, from the seed alone."""
    rng, dev = _rng(case, seed), "cuda"
    real_h = case["kind"] in ("fit", "md")  # the hydrogens' own LJ where forces are fitted or followed
    h = (SIG_H, EPS_H) if real_h else (0.0, 0.0)

    def water(n):
        L = float(np.float32((n / WATERS_PER_A3) ** (1.0 / 3.0)))
        x = _waters(rng, n, L, dev).reshape(-1, 3)
        return _system(_wrapped(x, L), np.tile([Q_O, Q_H, Q_H], n), np.tile([0, 1, 1], n), [SIG_O, h[0]],
                       [EPS_O, h[1]], L, _water_excl(n))

    if case["system"] == "lj":  # FCC sites with vacancies for sizes between, jittered
        n = case["atoms"]
        cells = max(4, math.ceil((n / 4) ** (1.0 / 3.0)))
        L = float(np.float32((max(n, 4 * 4 ** 3 * 0.9) / 0.0213) ** (1.0 / 3.0)))
        g = np.stack(np.meshgrid(*[np.arange(cells)] * 3, indexing="ij"), -1).reshape(-1, 1, 3)
        x = (g + np.array([[0, 0, 0], [.5, .5, 0], [.5, 0, .5], [0, .5, .5]])).reshape(-1, 3) * (L / cells)
        x = x[np.sort(rng.permutation(len(x))[:n])] + rng.uniform(-0.05, 0.05, (n, 3))
        return [_system(_wrapped(torch.from_numpy(x).to(dev), L), np.zeros(n), np.zeros(n), [3.4], [0.238], L,
                        np.zeros((0, 2)), cutoff=8.5, alpha=0.0)]
    if case["system"] == "chain":
        nc, nw = case["chain"], case["waters"]
        L = float(np.float32(((nc + 3 * nw) / CHAIN_ATOMS_PER_A3) ** (1.0 / 3.0)))
        chain = _chain(rng, nc, L)
        x = _waters(rng, nw, L, dev, torch.from_numpy(chain).to(dev)).reshape(-1, 3)
        x = torch.cat([torch.from_numpy(chain).to(dev), x])
        sig = rng.uniform(3.0, 4.0, 20) if real_h else rng.uniform(1.0, 4.0, 20)
        eps = rng.uniform(0.01, 0.2, 20)
        qc = rng.normal(0.0, 0.3, nc)
        i = np.arange(nc)
        excl = np.concatenate([np.stack([i[:-1], i[1:]], 1), np.stack([i[:-2], i[2:]], 1), _water_excl(nw, nc)])
        return [_system(_wrapped(x, L), np.concatenate([qc - qc.mean(), np.tile([Q_O, Q_H, Q_H], nw)]),
                        np.concatenate([rng.integers(0, 20, nc), np.tile([20, 21, 21], nw)]),
                        np.concatenate([sig, [SIG_O, h[0]]]), np.concatenate([eps, [EPS_O, h[1]]]), L, excl,
                        np.stack([i[:-3], i[3:]], 1))]
    if case.get("boxes", 1) == 1:
        return [water(case["waters"])]
    return [water(n) for n in _box_sizes(case)]


def _topology(s, nc):
    """Masses (hydrogens repartitioned to 4.032 amu), the chain's bonded terms and the rigid waters."""
    nw, i = (s.n_atoms - nc) // 3, np.arange(nc)
    mass = np.concatenate([np.full(nc, 12.011), np.tile([15.9994 + 2 * (1.008 - 4.032), 4.032, 4.032], nw)])
    nb_, na, nd = nc - 1, nc - 2, nc - 3
    return SimpleNamespace(
        mass=mass.astype(np.float32), bonds=np.stack([i[:-1], i[1:]], 1).astype(np.int32),
        bond_k=np.full(nb_, 300.0, np.float32), bond_r0=np.full(nb_, 1.5, np.float32),
        angles=np.stack([i[:-2], i[1:-1], i[2:]], 1).astype(np.int32), angle_k=np.full(na, 50.0, np.float32),
        angle_theta0=np.full(na, math.radians(111.0), np.float32),
        dihedrals=np.stack([i[:-3], i[1:-2], i[2:-1], i[3:]], 1).astype(np.int32),
        dihedral_k=np.full(nd, 0.2, np.float32), dihedral_n=np.full(nd, 3, np.int32),
        dihedral_phase=np.zeros(nd, np.float32),
        waters=(nc + 3 * np.arange(nw)[:, None] + np.arange(3)).astype(np.int32), water_roh=R_OH, water_rhh=R_HH)


def _velocities(case, seed, mass):
    rng = np.random.Generator(np.random.PCG64([902827, int(seed), 1]))
    return (rng.normal(size=(len(mass), 3)) * np.sqrt(0.0019872041 * 300.0 * 418.4 / mass)[:, None]).astype(np.float32)


def _fit_targets(case, seed, n, boxes):
    rng = np.random.Generator(np.random.PCG64([902827, int(seed), 2]))
    return rng.normal(0.0, 10.0, (n, 3)).astype(np.float32), rng.normal(0.0, 100.0, (boxes, 2))


def _pme_grid(s):
    """About one grid point per angstrom, a product of small primes (64 for the 62.2 A box)."""
    k = 2 * math.ceil(float(s.box[0]) / 2)
    while (2 ** 10 * 3 ** 6 * 5 ** 4) % k:
        k += 2
    return (k, k, k)


def prepare(case, seed):
    systems = _systems(case, seed)
    st = SimpleNamespace(case=case)
    st.pos, st.q, st.typ = nb.concat_inputs(systems)
    if case["kind"] == "noalloc":
        st.system = systems[0]
        st.F = torch.empty_like(st.pos)
        st.E = torch.empty(2, dtype=torch.float64, device="cuda")
        st.W = torch.empty(6, dtype=torch.float64, device="cuda")
        return st
    st.ctx = nb.Nonbonded(systems if len(systems) > 1 else systems[0])
    if case["option"] == "pme":
        st.ctx.set_pme(_pme_grid(systems[0]), 4)
    if case["option"] == "tables":
        st.ctx.set_tables(TABLE_N)
    if case["option"] == "host":
        st.pos, st.q, st.typ = (t.cpu().pin_memory() for t in (st.pos, st.q, st.typ))
        st.F = torch.empty(st.pos.shape, dtype=torch.float32, pin_memory=True)
        st.E = torch.empty((1, 2), dtype=torch.float64, pin_memory=True)
        st.W = torch.empty((1, 6), dtype=torch.float64, pin_memory=True)
    if case["kind"] == "fit":
        ft, et = _fit_targets(case, seed, len(st.pos), len(systems))
        st.ft, st.et = torch.from_numpy(ft).cuda(), torch.from_numpy(et).cuda()
        st.sigma = torch.from_numpy(systems[0].sigma.copy()).cuda().requires_grad_()
        st.eps = torch.from_numpy(systems[0].epsilon.copy()).cuda().requires_grad_()
        st.pos.requires_grad_()
        st.q.requires_grad_()
    if case["kind"] == "md":
        top = _topology(systems[0], case["chain"])
        st.ctx.md_init(top, **MD)
        st.vel = torch.from_numpy(_velocities(case, seed, top.mass)).cuda()
    return st


# --------------------------------------------------------------------- calls


def _loss(F, E, ft, et):
    """Force matching with the energies beside it."""
    return (F - ft).square().sum() / F.shape[0] + 1e-6 * (E - et).square().sum()


def run(st):
    kind = st.case["kind"]
    if kind == "noalloc":
        nb.forces_noalloc(st.system, st.pos, st.q, st.typ, st.F, st.E, st.W)
        return [st.F, st.E, st.W]
    if kind == "md":
        st.ctx.md_step(st.pos, st.vel, st.q, st.typ, n_steps=MD_STEPS)
        return [st.pos, st.vel]
    if kind == "fit":
        F, E = nb.nonbonded(st.pos, st.q, st.sigma, st.eps, st.ctx, st.typ)
        grads = torch.autograd.grad(_loss(F, E, st.ft, st.et), [st.pos, st.q, st.sigma, st.eps])
        with torch.no_grad():
            st.sigma -= FIT_RATE * grads[2].sign()
            st.eps -= FIT_RATE * grads[3].sign()
        return [F.detach(), E.detach(), *grads]
    if st.case["option"] == "host":
        return list(st.ctx.step(st.pos, st.q, st.typ, F=st.F, energy=st.E, virial=st.W))
    return list(st.ctx.step(st.pos, st.q, st.typ))


def work(case):
    """Bytes: the inputs (x, q, type and, for the adjoint and the dynamics, dL/dF or v) read once and the
    outputs written once.  Operations: 73 per unique pair inside the cutoff for the forces and energies (LJ
    with its switch, Ewald, both atoms' force sums), 163 more for their adjoint; PME: 64-point spread and
    gather (2 and 8 per point) and two real transforms of the grid."""
    if case["system"] == "lj":
        sizes, rho, rc = [case["atoms"]], 0.0213, 8.5
    elif case["system"] == "chain":
        sizes, rho, rc = [case["chain"] + 3 * case["waters"]], CHAIN_ATOMS_PER_A3, 9.0
    else:
        rho, rc, b = 3 * WATERS_PER_A3, 9.0, case.get("boxes", 1)
        if b == 1:
            sizes = [3 * case["waters"]]
        else:
            sizes = [3 * n for n in _box_sizes(case)]
    n = sum(sizes)
    pairs = 0.5 * n * rho * 4.0 / 3.0 * math.pi * rc ** 3
    nbytes, flops = n * (12 + 4 + 4 + 12) + 64 * len(sizes), 73.0 * pairs
    if case["kind"] == "fit":
        nbytes += n * (12 + 12 + 4)
        flops += 163.0 * pairs
    if case["option"] == "pme":
        k3 = n / rho
        flops += n * 64 * 10 + 2 * 2.5 * k3 * math.log2(k3)
    if case["kind"] == "md":
        nbytes, flops = MD_STEPS * n * (2 * 24 + 8 + 4), MD_STEPS * flops
    return {"bytes": float(nbytes), "flops": float(flops)}


# --------------------------------------------------- the same results in FP64


def _lj_tables(sigma, eps):
    s = 0.5 * (sigma[:, None] + sigma[None])
    e = torch.sqrt(eps[:, None] * eps[None])
    return 4.0 * e * s ** 12, 4.0 * e * s ** 6


def _candidate_pairs(x, L, rc):
    """Unique pairs (i, j) inside the cutoff, in chunks."""
    n, dev = len(x), x.device
    if n <= 40000:
        for i0 in range(0, n, 2048):
            m = min(2048, n - i0)
            r2 = _image(x[i0:i0 + m, None, 0] - x[None, i0:, 0], L).square()
            for a in (1, 2):
                r2 += _image(x[i0:i0 + m, None, a] - x[None, i0:, a], L).square()
            i, j = torch.nonzero(r2 < rc * rc, as_tuple=True)
            k = j > i
            yield i[k] + i0, j[k] + i0
        return
    nc = int(L / (rc + 1e-6))
    c = (x / L * nc).long().clamp_(0, nc - 1)
    cid = (c[:, 0] * nc + c[:, 1]) * nc + c[:, 2]
    order = torch.argsort(cid, stable=True)
    count = torch.bincount(cid, minlength=nc ** 3)
    start = torch.cumsum(count, 0) - count
    cap = int(count.max())
    table = torch.full((nc ** 3, cap), -1, dtype=torch.int64, device=dev)
    table[cid[order], torch.arange(n, device=dev) - start[cid[order]]] = order
    cells = torch.stack(torch.meshgrid(*[torch.arange(nc, device=dev)] * 3, indexing="ij"), -1).reshape(-1, 3)
    half = [(a, b, d) for a in (-1, 0, 1) for b in (-1, 0, 1) for d in (-1, 0, 1) if (a, b, d) >= (0, 0, 0)]
    per = max(1, 60_000_000 // (cap * cap))
    for o in half:
        nbr = (cells + torch.tensor(o, device=dev)) % nc
        nid = (nbr[:, 0] * nc + nbr[:, 1]) * nc + nbr[:, 2]
        for k0 in range(0, nc ** 3, per):
            ti, tj = table[k0:k0 + per], table[nid[k0:k0 + per]]
            r2 = _image(x[ti][:, :, None] - x[tj][:, None], L).square().sum(-1)
            ok = (r2 < rc * rc) & (ti >= 0)[:, :, None] & (tj >= 0)[:, None]
            if o == (0, 0, 0):
                ok &= ti[:, :, None] < tj[:, None]
            g, a, b = torch.nonzero(ok, as_tuple=True)
            yield ti[g, a], tj[g, b]


def _topology_pairs(s, dev):
    """(i, j, weight minus one of LJ and of Coulomb) of the excluded and the scaled pairs."""
    ex, p14 = torch.from_numpy(s.excl).long().to(dev), torch.from_numpy(s.pairs14).long().to(dev)
    ij = torch.cat([ex, p14])
    s_lj, s_c = float(np.float32(s.scale14_lj)), float(np.float32(s.scale14_coul))
    wl = torch.cat([torch.full((len(ex),), -1.0), torch.full((len(p14),), s_lj - 1.0)]).double().to(dev)
    wc = torch.cat([torch.full((len(ex),), -1.0), torch.full((len(p14),), s_c - 1.0)]).double().to(dev)
    return ij[:, 0], ij[:, 1], wl, wc


def _pair_chunks(s, x):
    """(i, j, w_lj, w_c): every pair inside the cutoff with weight 1, then what the excluded and scaled ones take back."""
    L, rc = float(s.box[0]), float(np.float32(s.cutoff))
    for i, j in _candidate_pairs(x, L, rc):
        yield i, j, 1.0, 1.0
    i, j, wl, wc = _topology_pairs(s, x.device)
    if len(i):
        k = _image(x[i] - x[j], L).square().sum(-1) < rc * rc
        yield i[k], j[k], wl[k], wc[k]


def _radial(s, r):
    """E12, E6, Ec and -r dE/dr of each, at r."""
    rc, rs, al = (float(np.float32(v)) for v in (s.cutoff, s.switch_dist, s.ewald_alpha))
    r2, den = r * r, (rc * rc - rs * rs) ** 3
    sw = r2 > rs * rs
    S = torch.where(sw, (rc * rc - r2) ** 2 * (rc * rc + 2 * r2 - 3 * rs * rs) / den, torch.ones_like(r))
    rS = torch.where(sw, 12 * r2 * (rc * rc - r2) * (rs * rs - r2) / den, torch.zeros_like(r))
    i6 = r2 ** -3
    ec = torch.erfc(al * r) / r
    fc = ec + 2 * al / math.sqrt(math.pi) * torch.exp(-al * al * r2)
    return S * i6 * i6, S * i6, ec, (12 * S - rS) * i6 * i6, (6 * S - rS) * i6, fc


def _short_range(s, x, q, typ, sigma, eps, tables=0):
    """F [N, 3], E [2], W [6]."""
    L, ke, rc = float(s.box[0]), float(np.float32(s.coulomb_k)), float(np.float32(s.cutoff))
    A, B = _lj_tables(sigma, eps)
    F, E, W = torch.zeros_like(x), x.new_zeros(2), x.new_zeros(6)
    for i, j, wl, wc in _pair_chunks(s, x):
        d = _image(x[i] - x[j], L)
        r2 = d.square().sum(-1)
        r = r2.sqrt()
        if tables:
            h = rc / tables
            k = (r / h).long().clamp_(0, tables - 1)
            lo, hi, t = _radial(s, k * h), _radial(s, (k + 1) * h), r / h - k
            e12, e6, ec, f12, f6, fc = (a + t * (b - a) for a, b in zip(lo, hi))
        else:
            e12, e6, ec, f12, f6, fc = _radial(s, r)
        a, b, qq = A[typ[i], typ[j]], B[typ[i], typ[j]], ke * q[i] * q[j]
        E[0] += (wl * (a * e12 - b * e6)).sum()
        E[1] += (wc * qq * ec).sum()
        f = ((wl * (a * f12 - b * f6) + wc * qq * fc) / r2)[:, None] * d
        F.index_add_(0, i, f)
        F.index_add_(0, j, f, alpha=-1.0)
        W += torch.stack([(d[:, u] * f[:, v]).sum() for u, v in ((0, 0), (1, 1), (2, 2), (0, 1), (0, 2), (1, 2))])
    return F, E, W


def _bspline(x, n):
    if n == 2:
        return torch.clamp(1.0 - (x - 1.0).abs(), min=0.0)
    return (x * _bspline(x, n - 1) + (n - x) * _bspline(x - 1.0, n - 1)) / (n - 1)


def _long_range(s, x, q, K, n=4):
    """Smooth PME with the self term and the corrections of the excluded and scaled pairs: F, E, W [6]."""
    dev, L = x.device, float(s.box[0])
    al, ke = float(np.float32(s.ewald_alpha)), float(np.float32(s.coulomb_k))
    u = x / L * K
    fl = u.floor()
    j = torch.arange(n, device=dev)
    idx = (fl[:, :, None].long() - j) % K
    arg = (u - fl)[:, :, None] + j
    w, dw = _bspline(arg, n), (_bspline(arg, n - 1) - _bspline(arg - 1.0, n - 1)) * (K / L)
    at = ((idx[:, 0, :, None, None] * K + idx[:, 1, None, :, None]) * K + idx[:, 2, None, None, :])
    prod = lambda a, b, c: a[:, :, None, None] * b[:, None, :, None] * c[:, None, None, :]  # noqa: E731
    Q = x.new_zeros(K ** 3)
    Q.index_add_(0, at.reshape(-1), (q[:, None, None, None] * prod(w[:, 0], w[:, 1], w[:, 2])).reshape(-1))
    FQ = torch.fft.fftn(Q.reshape(K, K, K))
    m = torch.fft.fftfreq(K, 1.0 / K, dtype=torch.float64, device=dev) / L
    mv = torch.meshgrid(m, m, m, indexing="ij")
    m2 = mv[0] ** 2 + mv[1] ** 2 + mv[2] ** 2
    m2[0, 0, 0] = 1.0
    k = torch.arange(n - 1, dtype=torch.float64, device=dev)
    ph = torch.exp(2j * math.pi * torch.outer(m * L, k) / K)
    mod = 1.0 / (ph * _bspline(k + 1.0, n)).sum(1).abs() ** 2
    G = ke * torch.exp(-math.pi ** 2 * m2 / al ** 2) / (math.pi * L ** 3 * m2) * (
        mod[:, None, None] * mod[None, :, None] * mod[None, None, :])
    G[0, 0, 0] = 0.0
    Em = 0.5 * G * FQ.abs() ** 2
    th = (torch.fft.ifftn(G * FQ).real * K ** 3).reshape(-1)[at]
    F = torch.stack([-q * (prod(dw[:, 0], w[:, 1], w[:, 2]) * th).sum((1, 2, 3)),
                     -q * (prod(w[:, 0], dw[:, 1], w[:, 2]) * th).sum((1, 2, 3)),
                     -q * (prod(w[:, 0], w[:, 1], dw[:, 2]) * th).sum((1, 2, 3))], 1)
    c = 2.0 * (1.0 + math.pi ** 2 * m2 / al ** 2) / m2
    W = torch.stack([(Em * ((1.0 if a == b else 0.0) - c * mv[a] * mv[b])).sum()
                     for a, b in ((0, 0), (1, 1), (2, 2), (0, 1), (0, 2), (1, 2))])
    E = Em.sum() - ke * al / math.sqrt(math.pi) * q.square().sum()
    i, k2, _, wc = _topology_pairs(s, dev)
    d = _image(x[i] - x[k2], L)
    r = d.norm(dim=1)
    qq, er = wc * ke * q[i] * q[k2], torch.erf(al * r)
    E = E + (qq * er / r).sum()
    f = (qq * (er / r - 2 * al / math.sqrt(math.pi) * torch.exp(-(al * r) ** 2)) / r ** 2)[:, None] * d
    F.index_add_(0, i, f)
    F.index_add_(0, k2, f, alpha=-1.0)
    W = W + torch.stack([(d[:, a] * f[:, b]).sum() for a, b in ((0, 0), (1, 1), (2, 2), (0, 1), (0, 2), (1, 2))])
    return F, E, W


def _bonded(t, x, L):
    """Forces of the chain's bonds, angles and dihedrals."""
    with torch.enable_grad():
        y = x.detach().requires_grad_()
        par = {k: torch.from_numpy(getattr(t, k)).to(x.device).double()
               for k in ("bond_k", "bond_r0", "angle_k", "angle_theta0", "dihedral_k", "dihedral_n", "dihedral_phase")}
        at = {k: torch.from_numpy(getattr(t, k)).to(x.device).long() for k in ("bonds", "angles", "dihedrals")}
        im = lambda a, b: _image(y[b] - y[a], L)  # noqa: E731
        b = at["bonds"]
        U = (par["bond_k"] * (im(b[:, 0], b[:, 1]).norm(dim=1) - par["bond_r0"]) ** 2).sum()
        a = at["angles"]
        p, q = im(a[:, 1], a[:, 0]), im(a[:, 1], a[:, 2])
        th = torch.atan2(torch.linalg.cross(p, q).norm(dim=1), (p * q).sum(1))
        U = U + (par["angle_k"] * (th - par["angle_theta0"]) ** 2).sum()
        d = at["dihedrals"]
        b1, b2, b3 = im(d[:, 0], d[:, 1]), im(d[:, 1], d[:, 2]), im(d[:, 2], d[:, 3])
        n1, n2 = torch.linalg.cross(b1, b2), torch.linalg.cross(b2, b3)
        phi = torch.atan2(b2.norm(dim=1) * (b1 * n2).sum(1), (n1 * n2).sum(1))
        U = U + (par["dihedral_k"] * (1 + torch.cos(par["dihedral_n"] * phi - par["dihedral_phase"]))).sum()
        return -torch.autograd.grad(U, y)[0]


def _normals(n, step, stream, seed):
    """Three normals per atom: Philox4x32-10 (Salmon et al. 2011) on (atom, step, stream, 0), 24-bit uniforms,
    Box-Muller."""
    M = np.uint64(0xFFFFFFFF)
    c = [np.arange(n, dtype=np.uint64), np.full(n, step, np.uint64), np.full(n, stream, np.uint64),
         np.zeros(n, np.uint64)]
    k = [seed & 0xFFFFFFFF, seed >> 32]
    for _ in range(10):
        p, r = np.uint64(0xD2511F53) * c[0], np.uint64(0xCD9E8D57) * c[2]
        c = [(r >> np.uint64(32)) ^ c[1] ^ np.uint64(k[0]), r & M, (p >> np.uint64(32)) ^ c[3] ^ np.uint64(k[1]), p & M]
        k = [(k[0] + 0x9E3779B9) & 0xFFFFFFFF, (k[1] + 0xBB67AE85) & 0xFFFFFFFF]
    u = [((v >> np.uint64(8)).astype(np.float64) + 0.5) * 2.0 ** -24 for v in c]
    a, b = np.sqrt(-2 * np.log(u[0])), np.sqrt(-2 * np.log(u[2]))
    return torch.from_numpy(np.stack([a * np.cos(2 * np.pi * u[1]), a * np.sin(2 * np.pi * u[1]),
                                      b * np.cos(2 * np.pi * u[3])], 1)).cuda()


def _dynamics(case, seed, s):
    """Positions and velocities after the steps of one call."""
    t = _topology(s, case["chain"])
    f32 = lambda v: float(np.float32(v))  # noqa: E731
    dt, L, dev = f32(MD["dt"]), float(s.box[0]), "cuda"
    x, q = torch.from_numpy(s.pos).to(dev).double(), torch.from_numpy(s.q).to(dev).double()
    typ = torch.from_numpy(s.type).to(dev).long()
    sigma, eps = (torch.from_numpy(p).to(dev).double() for p in (s.sigma, s.epsilon))
    m = torch.from_numpy(t.mass).to(dev).double()[:, None]
    v = torch.from_numpy(_velocities(case, seed, t.mass)).to(dev).double()
    c = math.exp(-f32(MD["gamma"]) * dt / 2)
    sg = torch.sqrt((1 - c * c) * 0.0019872041 * f32(MD["temperature"]) * 418.4 / m)
    w = torch.from_numpy(t.waters).to(dev).long()
    ca, cb = torch.tensor([0, 0, 1], device=dev), torch.tensor([1, 2, 2], device=dev)
    sign = torch.zeros(3, 3, dtype=torch.float64, device=dev)  # [atom, constraint]
    sign[ca, torch.arange(3)], sign[cb, torch.arange(3)] = 1.0, -1.0
    im = 1.0 / m[w][..., 0]
    C = sign[ca][None] * im[:, ca, None] - sign[cb][None] * im[:, cb, None]
    roh, rhh = f32(R_OH), f32(R_HH)
    d2 = torch.tensor([roh * roh, roh * roh, rhh * rhh], dtype=torch.float64, device=dev)

    def force(y):
        y = torch.remainder(y, L)
        F = _short_range(s, y, q, typ, sigma, eps)[0] + _bonded(t, y, L)
        return F + _long_range(s, y, q, _pme_grid(s)[0])[0]

    F = force(x)
    for step in range(MD_STEPS):
        v = c * v + sg * _normals(len(x), step, 0, MD["seed"])
        v = v + 0.5 * dt * 418.4 * F / m
        y = x + dt * v
        r, u = _image(x[w[:, ca]] - x[w[:, cb]], L), _image(y[w[:, ca]] - y[w[:, cb]], L)
        lam = torch.zeros(len(w), 3, dtype=torch.float64, device=dev)
        for _ in range(12):
            rr = u + torch.einsum("wkl,wl,wlc->wkc", C, lam, r)
            g = rr.square().sum(-1) - d2
            lam = lam - torch.linalg.solve(2 * C * torch.einsum("wkc,wlc->wkl", rr, r), g)
        move = torch.einsum("il,wl,wlc,wi->wic", sign, lam, r, im)
        y[w], v[w] = y[w] + move, v[w] + move / dt
        x, F = y, force(y)
        v = v + 0.5 * dt * 418.4 * F / m
        v = c * v + sg * _normals(len(x), step, 1, MD["seed"])
        r, dv = _image(x[w[:, ca]] - x[w[:, cb]], L), v[w[:, ca]] - v[w[:, cb]]
        mu = torch.linalg.solve(C * torch.einsum("wkc,wlc->wkl", r, r), -(r * dv).sum(-1))
        v[w] = v[w] + torch.einsum("il,wl,wlc,wi->wic", sign, mu, r, im)
    return [torch.remainder(x, L), v]


def _fitted(case, seed, systems):
    """F, E and the gradients of the loss, by automatic differentiation of the pair energies."""
    dev = "cuda"
    ft, et = _fit_targets(case, seed, sum(s.n_atoms for s in systems), len(systems))
    ft, et = torch.from_numpy(ft).to(dev).double(), torch.from_numpy(et).to(dev)
    sigma, eps = (torch.from_numpy(p).to(dev).double().requires_grad_()
                  for p in (systems[0].sigma, systems[0].epsilon))
    A, B = _lj_tables(sigma, eps)
    n_all, Fs, Es, gx, gq, at = len(ft), [], [], [], [], 0
    parts = []
    for k, s in enumerate(systems):
        L, ke = float(s.box[0]), float(np.float32(s.coulomb_k))
        x = torch.from_numpy(s.pos).to(dev).double().requires_grad_()
        q = torch.from_numpy(s.q).to(dev).double().requires_grad_()
        typ = torch.from_numpy(s.type).to(dev).long()
        ch = [(i, j, wl * torch.ones(len(i), dtype=torch.float64, device=dev),
               wc * torch.ones(len(i), dtype=torch.float64, device=dev))
              for i, j, wl, wc in _pair_chunks(s, x.detach())]
        i, j, wl, wc = (torch.cat(c) for c in zip(*ch))
        r = _image(x[i] - x[j], L).norm(dim=1)
        rc, rs, al = (float(np.float32(p)) for p in (s.cutoff, s.switch_dist, s.ewald_alpha))
        S = torch.where(r > rs, (rc * rc - r * r) ** 2 * (rc * rc + 2 * r * r - 3 * rs * rs) /
                        (rc * rc - rs * rs) ** 3, torch.ones_like(r))
        e_lj = (wl * S * (A[typ[i], typ[j]] * r ** -12 - B[typ[i], typ[j]] * r ** -6)).sum()
        e_c = (wc * ke * q[i] * q[j] * torch.erfc(al * r) / r).sum()
        F = -torch.autograd.grad(e_lj + e_c, x, create_graph=True)[0]
        E = torch.stack([e_lj, e_c])
        loss = (F - ft[at:at + len(x)]).square().sum() / n_all + 1e-6 * (E - et[k]).square().sum()
        g = torch.autograd.grad(loss, [x, q, sigma, eps], retain_graph=k + 1 < len(systems))
        at += len(x)
        Fs.append(F.detach())
        Es.append(E.detach())
        gx.append(g[0])
        gq.append(g[1])
        parts.append(g[2:])
    return [torch.cat(Fs), torch.stack(Es), torch.cat(gx), torch.cat(gq), sum(p[0] for p in parts),
            sum(p[1] for p in parts)]


def exact(case, seed):
    systems = _systems(case, seed)
    if case["kind"] == "md":
        return _dynamics(case, seed, systems[0])
    if case["kind"] == "fit":
        return _fitted(case, seed, systems)
    out = []
    for s in systems:
        x, q = torch.from_numpy(s.pos).cuda().double(), torch.from_numpy(s.q).cuda().double()
        typ = torch.from_numpy(s.type).cuda().long()
        sigma, eps = (torch.from_numpy(p).cuda().double() for p in (s.sigma, s.epsilon))
        F, E, W = _short_range(s, x, q, typ, sigma, eps, TABLE_N if case["option"] == "tables" else 0)
        if case["option"] == "pme":
            F2, E2, W2 = _long_range(s, x, q, _pme_grid(s)[0])
            F, W = F + F2, W + W2
            E[1] += E2
        out.append((F, E, W))
    if case["kind"] == "noalloc":
        return list(out[0])
    return [torch.cat([o[0] for o in out]), torch.stack([o[1] for o in out]), torch.stack([o[2] for o in out])]
