"""The forward kernel's block shapes give the same bits: blocks of 4 warps at
80 registers (one small system), at 64 registers (many work units: the batch)
and blocks of 8 warps (a large type-pair table).  The FP32 sums of a work unit
do not depend on which warp takes it, so the tolerance is zero; sizes lie on
both sides of the line at four units per resident warp (about 39,000 atoms)."""

import dataclasses

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_0902_0827_gb300 import nb
from paper_0902_0827_gb300 import systems as S

pytestmark = pytest.mark.gpu


def _forces(systems):
    ctx = nb.Nonbonded(systems)
    pos, q, t = nb.concat_inputs(systems)
    ctx.build(pos)
    F, E, W = ctx.forces(pos, q, t)
    torch.cuda.synchronize()
    ctx.status()
    return F, E, W


def _padded(s, n_types):
    """The same system with unused types behind its own."""
    n = n_types - len(s.sigma)
    assert n >= 0
    return dataclasses.replace(s, sigma=np.append(s.sigma, np.full(n, 3.0, np.float32)).astype(np.float32),
                               epsilon=np.append(s.epsilon, np.full(n, 0.1, np.float32)).astype(np.float32))


@pytest.mark.parametrize("n_types", [2, 22, 27, 64])
@pytest.mark.parametrize("copies", [1, 10, 12, 13, 14, 16])
def test_every_block_shape_gives_the_bits_of_one_small_system(copies, n_types):
    s = S.water_box(n_waters=1001)
    F1, E1, W1 = _forces([s])
    F, E, W = _forces([_padded(s, n_types)] * copies)
    for k in range(copies):
        assert torch.equal(F[k * s.n_atoms:(k + 1) * s.n_atoms], F1)
        assert torch.equal(E[k], E1[0]) and torch.equal(W[k], W1[0])
