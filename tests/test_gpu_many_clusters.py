"""Systems whose exclusion-mask records are numbered beyond 24 bits (six per
cluster: from 2.8 million clusters, 22.4 million atoms, on): 23.4 million atoms
on a jittered lattice, checked in a block of the last columns, whose atoms'
self tiles, exclusions and 1-4 pairs have the highest records, against the
oracle on the block's surroundings (every neighbour of the checked atoms)."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
from paper_0902_0827_gb300 import nb
from paper_0902_0827_gb300 import systems as S

pytestmark = pytest.mark.gpu

M, A, RC = 286, np.float32(3.0), 6.0  # lattice points per axis, spacing, cutoff


@pytest.fixture(scope="module")
def lattice():
    rng = np.random.default_rng(17)
    i = np.arange(M, dtype=np.float32)
    pos = np.empty((M, M, M, 3), np.float32)
    pos[..., 0] = i[:, None, None]
    pos[..., 1] = i[None, :, None]
    pos[..., 2] = i[None, None, :]
    pos = (pos.reshape(-1, 3) + np.float32(0.5)) * A
    pos += rng.uniform(-0.3, 0.3, pos.shape).astype(np.float32)
    n = pos.shape[0]
    q = rng.normal(0, 0.3, n).astype(np.float32)
    L = float(M * A)
    # neighbours along z in the block: pairs (k, k + 1), excluded and 1-4 in turn
    lo, hi = (90.0, L - 24.0, 90.0), (150.0, L - 3.0, 120.0)
    near = np.nonzero(np.all((pos >= np.float32(lo)) & (pos < np.float32(hi)), axis=1))[0]
    z = near % M
    ex, p14 = near[z % 4 == 0], near[z % 4 == 2]
    s = S.System("lattice", pos, q, np.zeros(n, np.int32), np.array([2.6], np.float32), np.array([0.2], np.float32),
                 np.full(3, L, np.float32), np.stack([ex, ex + 1], 1).astype(np.int32),
                 np.stack([p14, p14 + 1], 1).astype(np.int32), cutoff=RC, switch_dist=5.0, ewald_alpha=0.4)
    # the surroundings as a system of their own (the same box and coordinates)
    lo2, hi2 = np.float32(lo) - np.float32(3.0), np.float32(hi) + np.float32(2.9)
    sub = np.nonzero(np.all((pos >= lo2) & (pos < hi2), axis=1))[0]
    of = np.full(n, -1, np.int64)
    of[sub] = np.arange(len(sub))

    def within(p):
        m = of[p]
        return m[(m >= 0).all(1)].astype(np.int32)

    small = S.System("block", pos[sub], q[sub], s.type[sub], s.sigma, s.epsilon, s.box, within(s.excl),
                     within(s.pairs14), cutoff=RC, switch_dist=5.0, ewald_alpha=0.4)
    Fo = oracle.forces(small, method="cells")[0]
    inner = np.all((pos[sub] >= lo2 + np.float32(RC)) & (pos[sub] < hi2 - np.float32(RC)), axis=1)
    assert inner.sum() > 500
    return s, sub[inner], Fo[inner]


@pytest.mark.parametrize("group", [1, 4, 8])
def test_records_beyond_24_bits(lattice, group):
    s, atoms, Fo = lattice
    ctx = nb.Nonbonded(s)
    ctx.set_tuning(group_clusters=group)
    F, E, W = ctx.step(*nb.concat_inputs([s]))
    torch.cuda.synchronize()
    ctx.status()
    perm, cs = ctx.debug_cells()
    clusters = np.nonzero(np.isin(perm, atoms))[0] // 8
    assert 6 * clusters.min() > 1 << 24
    F = F[torch.from_numpy(atoms).cuda()].double().cpu().numpy()
    assert np.linalg.norm(F - Fo) <= 5e-6 * np.linalg.norm(Fo)
