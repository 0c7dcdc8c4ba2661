"""Prefix sums where their launch changes over: one block, one and two passes of a cluster, three
launches.  The pair list of a row of touching boxes is known in closed form."""
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


@pytest.mark.parametrize("n", [1, 2, 4095, 4096, 4097, 8191, 32769, 65535, 65536, 65537, 131072, 131073, 300001])
def test_pairs_of_a_row_of_boxes(P, n):
    b = S._bodies(n)
    b["he"] = 0.25
    b["mass"] = 1.0
    k = np.arange(n)
    b["c"][:, 0] = 0.5 * (k % 400)           # rows of 400 boxes face to face, far apart
    b["c"][:, 1] = 1.0
    b["c"][:, 2] = 4.0 * (k // 400)
    g = P.Scene(S.Scene("rows", S.default_params(n_iter=1), b, S._bonds(0), 1))
    g.detect()
    pairs = g.pairs()
    i = k[:-1][(k[:-1] % 400) != 399]
    assert np.array_equal(pairs, np.stack([i, i + 1], 1))
    g.close()
