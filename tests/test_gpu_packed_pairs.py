"""The forward kernel's packed pair arithmetic (two pairs per lane) against
its scalar form (nb_debug_pair_terms), bit for bit: boxes of two to nine atoms
whose single interacting pair lies at a given distance, in either half of the
8 x 8 tile, with and without Ewald and the switch."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_0902_0827_gb300 import nb
from paper_0902_0827_gb300 import systems as S

pytestmark = pytest.mark.gpu

RADII = [0.9, 1.0, 1.9, 3.3, 5.01, 7.4999, 7.5, 7.5001, 8.2, 8.99, 8.9999]


def _pair_box(r, n_far, alpha, switch):
    """Two atoms at distance r along a skew direction and n_far atoms out of reach of everything, all in one
    box; the far atoms (lower z) push the pair through the slots of its clusters."""
    L = 80.0
    d = np.array([0.48, 0.6, 0.64])
    a = np.array([40.3, 40.1, 40.2])
    far = np.stack([np.full(n_far, 40.3), np.full(n_far, 40.1), 2.0 + 0.0 * np.arange(n_far)], 1)
    far[:, 0] = np.mod(40.3 + 10.0 * np.arange(n_far), L)
    pos = np.concatenate([far, [a, a + r * d]])
    q = np.concatenate([np.zeros(n_far), [0.417, -0.834]])
    t = np.concatenate([np.zeros(n_far), [1, 2]])
    return S.System("pair", S.wrap_canonical(pos, np.full(3, L)), q.astype(np.float32), t.astype(np.int32),
                    np.array([0.0, 3.1, 2.2], np.float32), np.array([0.0, 0.15, 0.08], np.float32),
                    np.full(3, L, np.float32), np.zeros((0, 2), np.int32), np.zeros((0, 2), np.int32), cutoff=9.0,
                    switch_dist=switch, ewald_alpha=alpha)


@pytest.mark.parametrize("alpha,switch", [(0.32, 7.5), (0.0, 7.5), (0.32, 20.0)])
@pytest.mark.parametrize("n_far", [0, 3, 7])
def test_packed_pair_equals_scalar_pair(alpha, switch, n_far):
    boxes = [_pair_box(r, n_far, alpha, switch) for r in RADII]
    ctx = nb.Nonbonded(boxes)
    pos, q, t = nb.concat_inputs(boxes)
    F, E, _ = ctx.step(pos, q, t)
    torch.cuda.synchronize()
    ctx.status()
    n = n_far + 2
    x = torch.cat([pos, q[:, None]], 1).reshape(len(boxes), n, 4)
    ty = t.reshape(len(boxes), n)
    # the kernel's i atom is the one of the lower sorted slot: both orders give the same energies and opposite forces
    out = ctx.debug_pair_terms(x[:, n - 2], x[:, n - 1], ty[:, n - 2], ty[:, n - 1]).cpu().numpy().astype(np.float64)
    inside = out[:, 2] < np.float32(9.0) * np.float32(9.0)
    want = np.where(inside[:, None], out[:, :2], 0.0)
    assert inside.any()
    assert np.array_equal(E.cpu().numpy(), np.rint(want * 2.0 ** 32) / 2.0 ** 32)
    Fp = F.reshape(len(boxes), n, 3).cpu().numpy()
    fj = np.rint(np.where(inside[:, None], out[:, 4:7], 0.0) * 2.0 ** 32) / 2.0 ** 32
    assert np.array_equal(Fp[:, n - 1], fj.astype(np.float32))
    assert np.array_equal(Fp[:, n - 2], (-fj).astype(np.float32))
    assert not Fp[:, :n - 2].any()
