"""The branches of the PME kernels that ordinary systems leave out: charges so
large that a spread contribution takes the wide fixed-point path (|v| >= 32),
excluded pairs beyond 2 / alpha (their energy in FP64), charges taken by atom
index (nb_pme_forces after nb_build_cells alone) and from the sorted arrays
(nb_step), grids whose tiles hold one row, order 8 with its smaller hit
batches.  Against the oracle's smooth PME and corrections, with the bounds of
test_gpu_pme.py: forces, reciprocal energy 5e-6, pair corrections 1e-6."""

import dataclasses

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle.ewald as ew
from paper_0902_0827_gb300 import nb
from paper_0902_0827_gb300 import systems as S

pytestmark = pytest.mark.gpu


def _system(big):
    s = S.water_box(n_waters=230)
    q = s.q.copy()
    if big:
        q[0], q[300] = 500.0, -500.0
    d = s.pos[3::3].astype(np.float64) - s.pos[0]
    d -= s.box * np.rint(d / s.box)
    far = 3 + 3 * np.nonzero((np.linalg.norm(d, axis=1) > 6.6) & (np.linalg.norm(d, axis=1) < 8.5))[0][:5]
    ex = np.concatenate([s.excl, np.stack([np.zeros_like(far), far], 1)]).astype(np.int32)
    return dataclasses.replace(s, q=q, excl=ex)


@pytest.mark.parametrize("grid,order,big", [((20, 20, 20), 4, False), ((20, 20, 20), 4, True), ((24, 18, 540), 4, False),
                                            ((22, 22, 22), 6, False), ((22, 22, 22), 6, True), ((20, 24, 20), 8, True)])
def test_against_the_oracle(grid, order, big):
    s = _system(big)
    ctx = nb.Nonbonded(s)
    ctx.set_pme(grid, order)
    pos, q, t = nb.concat_inputs([s])
    ctx.build(pos)
    F, E, _ = ctx.pme_forces(pos, q)
    torch.cuda.synchronize()
    ctx.status()
    Fr, Er, _ = ew.spme(s, grid, order)
    Fc, Es, Ep, _ = ew.ewald_corrections(s)
    Fo = Fr + Fc
    assert np.linalg.norm(F.double().cpu().numpy() - Fo) <= 5e-6 * np.linalg.norm(Fo)
    E = E.cpu().numpy()
    assert abs(E[0] - Er) <= 5e-6 * abs(Er)
    assert abs(E[1] - Es) <= 1e-10 * abs(Es)
    assert abs(E[2] - Ep) <= 1e-6 * abs(Ep)
    # the whole step: long-range part = step with PME minus step without
    F1, E1, _ = ctx.step(pos, q, t)
    F1, E1 = F1.double(), E1.clone()
    ctx.set_pme(None)
    F0, E0, _ = ctx.step(pos, q, t)
    torch.cuda.synchronize()
    ctx.status()
    d = (F1 - F0.double()).cpu().numpy()
    assert np.linalg.norm(d - Fo) <= 5e-6 * (np.linalg.norm(Fo) + np.linalg.norm(F0.double().cpu().numpy()))
    assert abs((E1 - E0)[0, 1].item() - (Er + Es + Ep)) <= 5e-6 * (abs(Er) + abs(Es) + abs(Ep))
