"""The routes of an MD step.  A call of n steps runs one kernel between two
evaluations (second half, next first half, binning); n calls of one step run
the halves as two kernels.  Where the half-steps do not bin (page-locked host
charges, more than 8,192 columns) the binning kernel runs by itself.  Same
arithmetic, fixed-point sums: positions, velocities and energies have the same
bits on every route (tolerance zero).  Chains of 203 atoms leave partial warps
of free atoms and of waters."""

import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_0902_0827_gb300 import nb
from paper_0902_0827_gb300 import systems as S

pytestmark = pytest.mark.gpu


def _chain():
    s = S.dhfr_chain_md(n_chain=203, n_waters=805, L=30.6)
    return s, S.md_topology(s, 203), (32, 32, 32)


def _many_columns():
    rng = np.random.default_rng(8)
    box = np.array([1200.0, 1200.0, 18.5], np.float32)
    n = 107001
    pos = S.wrap_canonical(rng.uniform(0, 1, (n, 3)) * box, box)
    s = S.System("gas", pos, rng.normal(0, 0.05, n).astype(np.float32), np.zeros(n, np.int32),
                 np.array([0.0], np.float32), np.array([0.0], np.float32), box, np.zeros((0, 2), np.int32),
                 np.zeros((0, 2), np.int32), cutoff=8.5, switch_dist=7.5, ewald_alpha=0.3)
    top = S.md_topology(s, n)
    none = np.zeros(0, np.float32)
    top.bonds, top.bond_k, top.bond_r0 = np.zeros((0, 2), np.int32), none, none
    top.angles, top.angle_k, top.angle_theta0 = np.zeros((0, 3), np.int32), none, none
    top.dihedrals = np.zeros((0, 4), np.int32)
    top.dihedral_k, top.dihedral_n, top.dihedral_phase = none, np.zeros(0, np.int32), none
    return s, top, None


def _run(s, top, grid, calls, start, host=False):
    ctx = nb.Nonbonded(s)
    if grid:
        ctx.set_pme(grid, 4)
    ctx.md_init(top, dt=0.0005, gamma=5.0, temperature=300.0, seed=9)
    _, q, t = nb.concat_inputs([s])
    pos, vel = start[0].clone(), start[1].clone()
    E = torch.empty(6, dtype=torch.float64, device="cuda")
    if host:
        q, t = q.cpu().pin_memory(), t.cpu().pin_memory()
    ctx._sync_stream()
    for n in calls:
        code = nb.lib().nb_md_step(ctx.h, *(ctypes.c_void_p(x.data_ptr()) for x in (pos, vel, q, t)), n,
                                   ctypes.c_void_p(E.data_ptr()))
        assert code == 0
    torch.cuda.synchronize()
    ctx.status()
    return pos, vel, E


@pytest.mark.parametrize("case", ["chain_pme", "chain", "many_columns"])
def test_every_route_gives_the_same_bits(case):
    s, top, grid = _many_columns() if case == "many_columns" else _chain()
    grid = grid if case == "chain_pme" else None
    pos = torch.from_numpy(s.pos).cuda()
    if case != "many_columns":
        ctx = nb.Nonbonded(s)
        ctx.md_init(top)
        _, q, t = nb.concat_inputs([s])
        ctx.md_minimize(pos, q, t, 100)
        ctx.status()
    start = pos, torch.from_numpy(S.initial_velocities(top, 300.0)).cuda()
    want = _run(s, top, grid, [7], start)
    for calls, host in (([1] * 7, False), ([3, 4], False), ([7], True), ([1] * 7, True)):
        for x, y in zip(_run(s, top, grid, calls, start, host), want):
            assert torch.equal(x, y), (calls, host)
