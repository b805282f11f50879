"""The unpack kernel (fixed-point forces to FP32, the virial's atom part in
integers).  In a system without periodic-image pairs the virial is
sum_atoms x (x) F alone, so it is compared with that sum in FP64 over the
returned forces: each force is the FP32 rounding of its fixed-point sum
(relative 2^-24) and each of the atoms' terms is rounded to the 2^-20 grid
(2^-21), which bounds the difference.  Sizes around the block and the warp,
several systems inside one warp, and coordinates on both sides of 2,048 A
(beyond it the terms take FP64)."""

import dataclasses

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_0902_0827_gb300 import nb
from paper_0902_0827_gb300 import systems as S

pytestmark = pytest.mark.gpu


def _droplet(n, L):
    """The first n atoms of a water box (cut waters keep the exclusions among them) in the middle of a box of edge L."""
    w = S.water_box(n_waters=203)
    ex = w.excl[(w.excl < n).all(1)]
    box = np.full(3, L, np.float32)
    pos = S.wrap_canonical(w.pos[:n].astype(np.float64) + 0.5 * L - 9.0, box)
    return dataclasses.replace(w, pos=pos, q=w.q[:n].copy(), type=w.type[:n].copy(), excl=ex, box=box)


def _check(systems):
    ctx = nb.Nonbonded(systems if len(systems) > 1 else systems[0])
    F, E, W = ctx.step(*nb.concat_inputs(systems))
    torch.cuda.synchronize()
    ctx.status()
    F, W, at = F.cpu().numpy().astype(np.float64), W.cpu().numpy(), 0
    for k, s in enumerate(systems):
        f, x = F[at:at + s.n_atoms], s.pos.astype(np.float64)
        at += s.n_atoms
        for c, (a, b) in enumerate(((0, 0), (1, 1), (2, 2), (0, 1), (0, 2), (1, 2))):
            bound = np.abs(x[:, a] * f[:, b]).sum() * 2.0 ** -24 + s.n_atoms * 2.0 ** -21 + 1e-9
            assert abs(W[k, c] - (x[:, a] * f[:, b]).sum()) <= bound
    assert s.n_atoms < 2 or np.abs(f).max() > 0.0 or s.n_atoms < 4


@pytest.mark.parametrize("n", [1, 2, 31, 33, 63, 64, 65, 128, 600])
def test_sizes(n):
    _check([_droplet(n, 60.0)])


def test_systems_within_a_warp():
    _check([_droplet(n, 60.0) for n in (5, 9, 1, 40, 3, 64, 7)])


@pytest.mark.parametrize("L", [2040.0, 4090.0, 4400.0])
def test_large_coordinates(L):
    _check([_droplet(300, L)])
