"""The list kernel of one-cluster groups against the general one: the pair
sets of groups of 1 and of 4 clusters are the same, and the forces agree to
FP32 rounding, where the walk of every second cluster and the partner map can
go wrong: columns of odd length, boxes whose windows cross a z image, few and
empty columns, several systems (odd group offsets), exclusions."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
from paper_0902_0827_gb300 import nb
from paper_0902_0827_gb300 import systems as S

pytestmark = pytest.mark.gpu


def _lj(n, box, seed):
    rng = np.random.default_rng(seed)
    box = np.asarray(box, np.float32)
    pos = S.wrap_canonical(rng.uniform(0, 1, (n, 3)) * box, box)
    # charges only: random positions may nearly coincide
    return S.System("gas", pos, rng.normal(0, 0.2, n).astype(np.float32), np.zeros(n, np.int32),
                    np.array([0.0], np.float32), np.array([0.0], np.float32), box, np.zeros((0, 2), np.int32),
                    np.zeros((0, 2), np.int32), cutoff=8.5, switch_dist=7.5, ewald_alpha=0.3)


def _droplets(n, L, seed):
    """Half of the atoms in one corner, the rest anywhere: long, short and empty columns."""
    s = _lj(n, (L, L, L), seed)
    s.pos[: n // 2] = s.pos[: n // 2] * 0.2
    return s


CASES = {
    "small_box": lambda: [_lj(333, (17.2, 17.2, 17.2), 1)],
    "flat": lambda: [_lj(700, (60.0, 17.5, 18.0), 2)],
    "tall": lambda: [_lj(901, (17.5, 18.0, 90.0), 3)],
    "one_column": lambda: [_lj(57, (30.0, 30.0, 30.0), 4)],
    "droplet": lambda: [_droplets(1500, 50.0, 5)],
    "batch": lambda: [_lj(n, (18.0, 19.0, 20.0), 7 + n) for n in (9, 130, 77, 401, 8, 250)],
    # above 8,192 columns: the binning kernel's scan instead of the column sort's own sums
    "many_columns": lambda: [_lj(107000, (1200.0, 1200.0, 18.5), 8)],
    "waters": lambda: [S.water_box(n_waters=n) for n in (199, 307, 512)],
}


@pytest.mark.parametrize("name", list(CASES))
def test_groups_of_one_and_four(name):
    systems = CASES[name]()
    got = {}
    for group in (1, 4):
        ctx = nb.Nonbonded(systems if len(systems) > 1 else systems[0])
        ctx.set_tuning(group_clusters=group, list_capacity=4096)
        F, E, W = ctx.step(*nb.concat_inputs(systems))
        torch.cuda.synchronize()
        ctx.status()
        pairs, n, n_eval = ctx.debug_pairs()
        assert n == n_eval == len(np.unique(pairs, axis=0))
        got[group] = (pairs, F.double().cpu().numpy())
    assert np.array_equal(got[1][0], got[4][0])
    F1, F4 = got[1][1], got[4][1]
    assert np.linalg.norm(F1 - F4) <= 5e-6 * np.linalg.norm(F4)
    if name == "many_columns":
        Fo, _, _, n_pairs = oracle.forces(systems[0], method="cells")
        assert n_pairs == len(got[1][0])
        assert np.linalg.norm(F1 - Fo) <= 5e-6 * np.linalg.norm(Fo)
