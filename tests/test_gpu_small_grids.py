"""The forward kernel on grids smaller than the SMs hold (blocks_per_sm 1 and 2):
block shapes of their own, on both sides of the line from which a full grid
takes the 64-register shape, direct and tabulated.  Which block takes which
work unit does not change any result: tolerance zero against the full grid."""

import pytest

torch = pytest.importorskip("torch")

from paper_0902_0827_gb300 import nb
from paper_0902_0827_gb300 import systems as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tables", [0, 1024])
@pytest.mark.parametrize("n_waters", [200, 1001, 20001])
def test_small_grids_give_the_bits_of_the_full_one(n_waters, tables):
    s = S.water_box(n_waters=n_waters)
    ctx = nb.Nonbonded(s)
    ctx.set_tables(tables)
    inp = nb.concat_inputs([s])
    want = None
    for blocks in (3, 1, 2, 4):
        ctx.set_tuning(blocks_per_sm=blocks)
        got = ctx.step(*inp)
        torch.cuda.synchronize()
        ctx.status()
        want = want or [x.clone() for x in got]
        for x, y in zip(got, want):
            assert torch.equal(x, y)
