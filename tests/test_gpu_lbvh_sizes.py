"""The LBVH's pair list equals the grid's (and brute force's) at the edges of its sort tiles, with
more partners than a body's stash holds, equal Morton codes, several groups and pinned bodies."""
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


def _cloud(n, side, groups=1, same=False):
    """n turned boxes of edge 0.4 to 1.2 in a cube of the given side; same: all at one place but
    for their order (equal codes)."""
    rng = np.random.default_rng(n)
    b = S._bodies(n)
    b["he"] = rng.uniform(0.2, 0.6, (n, 3))
    b["mass"] = 1.0
    b["c"] = rng.uniform(0.0, side, (n, 3)) if not same else 0.25
    b["quat"] = S._random_unit_quats(rng, n)
    b["pinned"][rng.random(n) < 0.2] = 1
    b["group"] = np.arange(n) * groups // n
    return S.Scene("cloud", S.default_params(n_iter=1, has_ground=0), b, S._bonds(0), 1)


@pytest.mark.parametrize("n,side,groups,same", [(1, 1.0, 1, False), (2, 0.5, 1, False), (3, 0.5, 1, False),
                                                (40, 0.3, 1, True), (100, 2.0, 3, False), (1023, 8.0, 1, False),
                                                (1024, 4.0, 1, False), (1025, 8.0, 4, False), (2049, 12.0, 1, False),
                                                (5000, 20.0, 7, False)])
def test_lbvh_pairs_equal_the_grids(P, n, side, groups, same):
    sc = _cloud(n, side, groups, same)
    lists = []
    for bp in (1, 0):
        g = P.Scene(sc, broadphase=bp, max_pairs=max(64, 200 * n), max_contacts=max(64, 800 * n))
        g.detect()
        lists.append(g.pairs())
        g.detect()
        assert np.array_equal(g.pairs(), lists[-1])
        g.close()
    assert np.array_equal(lists[0], lists[1])
    if same:
        free = np.asarray(sc.bodies["pinned"]) == 0
        i, j = np.triu_indices(n, 1)
        assert len(lists[0]) == np.count_nonzero(free[i] | free[j])
