"""A build that fails on the host between its binning and its list kernel: the
call reports the CUDA error, and the next build starts from zero column counts.
(With the counts of two builds every atom is staged twice, and the column sort
writes past its arrays: this test is only for a library that clears them.)

The failure is a real one without a fault: the PME streams of the context take
part in a capture on another stream, so that an eager call may bin its atoms
but not fork its PME chain.  Results after it are compared bit for bit with a
context that saw no failure (the sums are fixed point: tolerance zero)."""

import ctypes

import pytest

torch = pytest.importorskip("torch")

from paper_0902_0827_gb300 import nb
from paper_0902_0827_gb300 import systems as S

pytestmark = pytest.mark.gpu
RELAXED = 2
NB_ERR_CUDA, NB_ERR_NOT_BUILT = 3, 5


def _fresh(s, pos, q, t, group):
    ctx = nb.Nonbonded(s)
    ctx.set_tuning(group_clusters=group)
    ctx.set_pme((24, 24, 24), 4)
    out = [x.clone() for x in ctx.step(pos, q, t)]
    torch.cuda.synchronize()
    ctx.status()
    return out


@pytest.mark.parametrize("group", [1, 4])
@pytest.mark.parametrize("call", ["step", "md_step"])
def test_next_build_after_a_failed_one(call, group):
    cu = ctypes.CDLL("libcuda.so.1")
    s = S.water_box(n_waters=300)
    top = S.md_topology(s)
    pos, q, t = nb.concat_inputs([s])
    vel = torch.from_numpy(S.initial_velocities(top, 300.0)).cuda()
    ctx = nb.Nonbonded(s)
    ctx.set_tuning(group_clusters=group)
    ctx.set_pme((24, 24, 24), 4)
    ctx.md_init(top, dt=0.0005, gamma=1.0, temperature=300.0, seed=3)
    F = torch.empty_like(pos)
    E = torch.empty((1, 2), dtype=torch.float64, device="cuda")
    W = torch.empty((1, 6), dtype=torch.float64, device="cuda")
    a, b = torch.cuda.Stream(), torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.stream(b):
        ctx.md_step(pos, vel, q, t, 2)
        ctx.step(pos, q, t, F, E, W)
    torch.cuda.synchronize()
    assert cu.cuStreamBeginCapture_v2(ctypes.c_void_p(a.cuda_stream), RELAXED) == 0
    with torch.cuda.stream(a):
        ctx.step(pos, q, t, F, E, W)
    with torch.cuda.stream(b), pytest.raises(nb.NbError) as err:
        if call == "step":
            ctx.step(pos, q, t, F, E, W)
        else:
            ctx.md_step(pos, vel, q, t, 2)
    assert err.value.code == NB_ERR_CUDA
    graph = ctypes.c_void_p()
    assert cu.cuStreamEndCapture(ctypes.c_void_p(a.cuda_stream), ctypes.byref(graph)) != 0
    with torch.cuda.stream(b), pytest.raises(nb.NbError) as err:
        ctx.forces(pos, q, t, F, E, W)
    assert err.value.code == NB_ERR_NOT_BUILT
    torch.cuda.synchronize()
    ctx.status()
    # the same context, twice: the first build after the failure, and one after a whole one
    want = _fresh(s, pos, q, t, group)
    for _ in range(2):
        with torch.cuda.stream(b):
            got = ctx.step(pos, q, t, F, E, W)
        torch.cuda.synchronize()
        ctx.status()
        for x, y in zip(got, want):
            assert torch.equal(x, y)
