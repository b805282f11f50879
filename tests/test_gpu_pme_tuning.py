"""A step with PME under every tuning of the grid: the forward kernel's grid and
the list kernel of each group size leave room for the PME chain by rules of
their own, and which block takes which work unit does not change any result.
So for a given group size and list split the steps of all grids have the same
bits, those of a rebuild followed by the forces (tolerance zero: the sums are
fixed point), with a small type table and with one that takes blocks of 8
warps."""

import dataclasses

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_0902_0827_gb300 import nb
from paper_0902_0827_gb300 import systems as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_types", [2, 30])
@pytest.mark.parametrize("group", [1, 4, 8])
@pytest.mark.parametrize("split", [1, 4])
def test_every_grid_gives_the_same_step(group, split, n_types):
    s = S.water_box(n_waters=701)
    extra = n_types - len(s.sigma)
    s = dataclasses.replace(s, sigma=np.append(s.sigma, np.full(extra, 3.0, np.float32)).astype(np.float32),
                            epsilon=np.append(s.epsilon, np.full(extra, 0.1, np.float32)).astype(np.float32))
    ctx = nb.Nonbonded(s)
    ctx.set_pme((32, 32, 32), 4)
    pos, q, t = nb.concat_inputs([s])
    ctx.set_tuning(group_clusters=group, list_split=split)
    ctx.build(pos)
    want = [x.clone() for x in ctx.forces(pos, q, t)]
    for blocks in (1, 2, 3, 4, 8):
        ctx.set_tuning(blocks_per_sm=blocks)
        for _ in range(2):
            got = ctx.step(pos, q, t)
            torch.cuda.synchronize()
            ctx.status()
            for x, y in zip(got, want):
                assert torch.equal(x, y)


@pytest.mark.parametrize("n_waters,tables", [(18001, 1024), (25001, 1024), (45001, 0), (66667, 0)])
def test_both_sides_of_the_line_between_shared_and_full_grids(n_waters, tables):
    s = S.water_box(n_waters=n_waters)
    ctx = nb.Nonbonded(s)
    ctx.set_tables(tables)
    ctx.set_pme((64, 64, 64), 4)
    pos, q, t = nb.concat_inputs([s])
    ctx.build(pos)
    want = [x.clone() for x in ctx.forces(pos, q, t)]
    for _ in range(3):
        got = ctx.step(pos, q, t)
        torch.cuda.synchronize()
        ctx.status()
        for x, y in zip(got, want):
            assert torch.equal(x, y)
