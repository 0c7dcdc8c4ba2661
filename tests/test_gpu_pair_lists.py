"""Pairs of bodies with as many partners as the count lists, one more, and hundreds; in one cell, and
of bodies off the grid: equal to brute force, to the LBVH's and to the allocation-free call's."""
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


def _clusters(sizes, spread, fast=0):
    """Clusters of overlapping unit cubes of the given sizes, 10 apart, and far more boxes than the
    small front takes; `fast` of them so fast that they leave the grid."""
    n = sum(sizes) + 200
    rng = np.random.default_rng(n)
    b = S._bodies(n)
    b["he"], b["mass"] = 0.5, 1.0
    at = 0
    for k, m in enumerate(sizes):
        b["c"][at:at + m] = np.array([10.0 * k, 5.0, 0.0]) + rng.uniform(-spread, spread, (m, 3))
        at += m
    b["c"][at:] = np.array([0.0, 5.0, 30.0]) + 10.0 * np.stack([np.arange(200) % 20, np.zeros(200), np.arange(200) // 20], 1)
    b["v"][at:at + fast] = (900.0, 0.0, 0.0)
    return S.Scene("clusters", S.default_params(n_iter=1, has_ground=0), b, S._bonds(0), 1)


@pytest.mark.parametrize("sizes,spread,fast", [([2, 5, 6, 16, 17, 18], 0.1, 0), ([33, 34, 65, 66], 0.1, 3),
                                               ([40] * 30, 0.6, 0), ([300], 0.05, 1), ([17, 40, 90], 0.9, 5)])
def test_pair_lists_equal_brute_force(P, sizes, spread, fast):
    import torch
    sc = _clusters(sizes, spread, fast)
    n, b, p = sc.n_bodies, sc.bodies, sc.params
    f = np.float32
    infl = (f(p["d_hat_rel"]) * f(1.0) + f(p["h"]) * np.sqrt((b["v"].astype(f) ** 2).sum(1, dtype=f))) + f(p["margin"])
    e = f(0.5) + infl
    lo, hi = b["c"].astype(f) - e[:, None], b["c"].astype(f) + e[:, None]
    i, j = np.triu_indices(n, 1)
    ok = (lo[i] <= hi[j]).all(1) & (lo[j] <= hi[i]).all(1)
    want = np.stack([i[ok], j[ok]], 1)
    for bp in (0, 1):
        g = P.Scene(sc, broadphase=bp, max_pairs=400 * n, max_contacts=4000 * n)
        g.detect()
        assert np.array_equal(g.pairs(), want), bp
        g.close()
    q = np.zeros((n, 12), f)
    q[:, :3], q[:, 3], q[:, 7], q[:, 11] = b["c"], 1, 1, 1
    on = lambda a: torch.tensor(a, device="cuda")
    pad = lambda a: on(np.pad(a, ((0, 0), (0, 1))).astype(f))
    t = [on(q), pad(b["v"]), pad(b["he"]), on(b["group"].astype(np.int32)), on((b["pinned"] & 1).astype(np.int32))]
    for cap in (len(want) + 7, len(want) // 2):
        pairs = torch.full((cap + 8, 2), -7, dtype=torch.int32, device="cuda")
        cnt = torch.zeros(1, dtype=torch.int32, device="cuda")
        P.pabd_broadphase_noalloc(*[x.data_ptr() for x in t], n, p["h"], p["margin"], p["d_hat_rel"], pairs.data_ptr(),
                                  cap, cnt.data_ptr(), torch.cuda.current_stream().cuda_stream)
        torch.cuda.synchronize()
        assert int(cnt.item()) == len(want)
        got = pairs.cpu().numpy()
        assert (got[min(cap, len(want)):] == -7).all()
        if cap >= len(want):
            assert np.array_equal(got[:len(want)], want)
        else:
            key = got[:cap, 0].astype(np.int64) * n + got[:cap, 1]
            assert (np.diff(key) > 0).all() and np.isin(key, want[:, 0].astype(np.int64) * n + want[:, 1]).all()


@pytest.mark.parametrize("crowd,spread", [(3, 0.3), (30, 0.6), (60, 1.5)])
def test_pairs_across_levels(P, crowd, spread):
    """Boxes of the grid's three levels and wider, a few or many to a cell (more to a lane than the
    count keeps), some pinned: the oracle's pairs, from the grid and from the LBVH."""
    import oracle as O
    sc = _clusters([crowd] * 10, spread)
    b = sc.bodies
    rng = np.random.default_rng(crowd)
    for k, he in enumerate([2.5] * 12 + [9.0] * 5 + [60.0] * 2):
        b["he"][k] = he
        b["c"][k] = (rng.uniform(0, 90), 5.0 + rng.uniform(-he, he), rng.uniform(-he, he))
    b["pinned"][rng.integers(0, sc.n_bodies, 40)] = 1
    ref = O.OracleScene(sc)
    ref.detect()
    want = ref.pairs()
    assert len(want) > 10 * crowd
    for bp in (0, 1):
        g = P.Scene(sc, broadphase=bp, max_pairs=400 * sc.n_bodies, max_contacts=4000 * sc.n_bodies)
        g.detect()
        assert np.array_equal(g.pairs(), want), bp
        g.close()
