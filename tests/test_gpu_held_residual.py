"""The residual of a held group is that of its last step, or zero before its first: the trial sweeps of
the launch-shape tuner leave no trace in it."""
import numpy as np
import pytest

import scenes as S

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__ as g
    g.build()
    import paper_2609_02675_gb300 as mod
    return mod


def _groups(sizes):
    """Stacked piles of the given sizes as the groups of one scene."""
    bodies = []
    for g, n in enumerate(sizes):
        b = S.box_pile_n(n, seed=30 + g, stacked=True).bodies
        b["group"] = g
        bodies.append(b)
    return S.Scene("groups", S.box_pile_n(2, n_iter=6).params, np.concatenate(bodies), S._bonds(0), 1)


# groups in clusters, groups of a launch per sweep, small groups alone, one of more than a residual chunk
@pytest.mark.parametrize("sizes", [(130, 40, 200), (300, 900, 20), (20, 30, 9), (5000, 60, 4500)])
@pytest.mark.parametrize("mode", [0, 1, 2, 3])
def test_held_groups_residual(P, sizes, mode):
    g = P.Scene(_groups(sizes), sweep_mode=mode)
    g.set_group_hold([1, 0, 1])
    g.step(2)
    r = g.residual()
    assert r[0] == 0.0 and r[1] > 0.0 and r[2] == 0.0
    g.set_group_hold([0, 1, 1])
    g.step(1)
    r2 = g.residual()
    assert r2[0] > 0.0 and r2[1] == r[1] and r2[2] == 0.0
    g.set_group_hold(None)
    g.tune()
    g.set_group_hold([1, 1, 0])
    g.step(1)
    r3 = g.residual()
    assert r3[0] == r2[0] and r3[1] == r[1] and r3[2] > 0.0
    g.close()
