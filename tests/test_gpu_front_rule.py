"""Small crowded scenes on both sides of the rule by which a step starts with the one-launch front: it is
left out where the state has many contacts, at creation and when the scene is tuned again, and the
states are those of the same bodies beside a group that makes the scene too large for it."""
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


def _crowd(n, side):
    rng = np.random.default_rng(n)
    b = S._bodies(n)
    b["he"], b["mass"] = 0.5, 1.0
    b["c"] = rng.uniform(0.0, side, (n, 3)) + 1.0
    b["quat"] = S._random_unit_quats(rng, n)
    b["pinned"][::17] = 1
    return b


def _nodes(g):
    return g.info()["graph_nodes"]


# a few contacts to a body, near the rule's line from both sides (bodies with more than 64 bond ends
# in the front's block), far beyond it
@pytest.mark.parametrize("n,side", [(40, 6.0), (40, 2.5), (128, 4.0), (60, 2.0), (100, 2.0), (60, 1.0), (128, 1.2)])
@pytest.mark.parametrize("mode", [1, 2])
def test_crowds_step_alike(P, n, side, mode):
    outs, heavy = [], []
    for extra in (0, 120):
        b = [_crowd(n, side)]
        if extra:
            far = S._bodies(extra)
            far["he"], far["mass"], far["group"] = 0.5, 1.0, 1
            far["c"][:, 0], far["c"][:, 1] = 5.0 * np.arange(extra), 3.0
            b.append(far)
        sc = S.Scene("crowd", S.default_params(n_iter=2), np.concatenate(b), S._bonds(0), 1)
        g = P.Scene(sc, sweep_mode=mode, sweep_lanes=16, light_order=1, max_pairs=20000, max_contacts=100000)
        g.step(1)
        i = g.info()
        assert (i["graph_nodes"] < 12) == (extra == 0 and i["n_contacts"] <= 1024), i["n_contacts"]
        heavy.append(i["heavy_bodies"])
        g.step_eager(1)
        outs.append((g.state()[:n], g.residual()[:1]))
        g.close()
    assert heavy[0] == heavy[1]
    assert all(np.array_equal(x, y) for x, y in zip(*outs))


def test_tuning_again_chooses_the_front_anew(P):
    crowd, apart = _crowd(100, 2.0), _crowd(100, 40.0)
    sc = S.Scene("crowd", S.default_params(n_iter=2), crowd, S._bonds(0), 1)
    cap = dict(max_pairs=20000, max_contacts=100000)
    g = P.Scene(sc, **cap)
    s0, n0 = g.state(), _nodes(g)
    h = P.Scene(S.Scene("apart", sc.params, apart, S._bonds(0), 1), **cap)
    s1, n1 = h.state(), _nodes(h)
    assert n0 > 12 > n1
    g.set_state(s1)
    g.tune()
    assert _nodes(g) < 12
    h.set_state(s0)
    h.tune()
    assert _nodes(h) > 12
    for x, y in ((g, h), (h, g)):
        x.set_state(s1 if x is g else s0)
        y.set_state(s1 if x is g else s0)
        x.step(2)
        y.step(2)
        assert np.array_equal(x.state(), y.state())
    g.close()
    h.close()
