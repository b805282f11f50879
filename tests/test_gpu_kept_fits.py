"""The fits of the Ewald factors are kept for the last alpha rc: nb_forces_noalloc
that goes from one product to another and back, and contexts created by several
threads at once, get the results of a context of their own (tolerance zero)."""

import dataclasses
import threading

import pytest

torch = pytest.importorskip("torch")

from paper_0902_0827_gb300 import nb
from paper_0902_0827_gb300 import systems as S

pytestmark = pytest.mark.gpu
ALPHAS = (0.32, 0.30, 0.32, 0.32, 0.35, 0.30)


def _step(s, inp):
    ctx = nb.Nonbonded(s)
    F = ctx.step(*inp)[0].clone()
    torch.cuda.synchronize()
    ctx.status()
    return F


def test_alternating_products():
    base = S.water_box(n_waters=250)
    inp = nb.concat_inputs([base])
    systems = {a: dataclasses.replace(base, ewald_alpha=a) for a in ALPHAS}
    want = {a: _step(s, inp) for a, s in systems.items()}
    assert not torch.equal(want[0.32], want[0.30])
    for a in ALPHAS:
        F = torch.empty_like(inp[0])
        nb.forces_noalloc(systems[a], *inp, F)
        assert torch.equal(F, want[a]), a
    got = {}

    def work(k):
        with torch.cuda.stream(torch.cuda.Stream()):
            got[k] = [_step(systems[a], inp) for a in ALPHAS[k % 2:] * 3]

    torch.cuda.synchronize()
    threads = [threading.Thread(target=work, args=(k,)) for k in range(4)]
    for th in threads:
        th.start()
    for th in threads:
        th.join()
    for k in range(4):
        for a, F in zip(ALPHAS[k % 2:] * 3, got[k]):
            assert torch.equal(F, want[a])
