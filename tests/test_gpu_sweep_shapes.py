"""The sweep's launch shapes at the sizes where they change over: the launch of all sweeps over
clusters of small groups, the launches per sweep with a thread per lane and per two lanes, and
the cooperative sweep give the same states bit for bit, and agree with the oracle."""
import numpy as np
import pytest

import oracle as O
import scenes as S
from gpu_helpers import REL_TOL, rel_err, teacher_forced_step

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


def _pile(n):
    return S.box_pile_n(n, stacked=True, n_iter=7)


def _groups(sizes):
    """Stacked piles of the given sizes as the groups of one scene, the first box pinned."""
    bodies = []
    for g, n in enumerate(sizes):
        b = _pile(n).bodies
        b["group"] = g
        bodies.append(b)
    sc = S.Scene("groups", _pile(sizes[0]).params, np.concatenate(bodies), S._bonds(0), 1)
    sc.bodies["pinned"][0] = 1
    return sc


# a group that fills its cluster's threads exactly, one body fewer and more (16 lanes: 256
# bodies; 4 lanes: 1024), one-body groups, groups that do not fill a block, more clusters than
# the device holds; a body with 400 ends and one with 100 inside a cluster; odd and even sweeps
SMALL = [(lambda: _pile(256), 16), (lambda: _pile(255), 16), (lambda: _pile(257), 16), (lambda: _pile(1024), 4),
         (lambda: _groups([1] * 9 + [3, 2]), 16), (lambda: _groups([130, 7, 40, 129]), 16),
         (lambda: _groups([200] * 12), 16), (lambda: _groups([33, 31]), 2), (lambda: _groups([5, 9]), 1),
         (lambda: S.slab_pile(10), 16), (lambda: S.slab_pile(5), 16), (lambda: S.chain_pendulum(), 16),
         (lambda: S.mass_ratio_chain(n=9), 16), (lambda: S.batched_trees(n_scenes=5), 16)]
# more lanes than the device's threads: two lanes per thread (and bodies on the extended path)
LARGE = [(lambda: _pile(4865), 16), (lambda: _pile(19501), 4), (lambda: _pile(40001), 2),
         (lambda: S.quadruped_bed_rod(bed=(32, 5, 32)), 16)]


@pytest.mark.parametrize("make,lanes", SMALL + LARGE)
def test_launch_shapes_bit_identical(P, make, lanes):
    outs = []
    for mode in (2, 1, 3):
        sc = make()
        g = P.Scene(sc, sweep_mode=mode, sweep_lanes=lanes)
        g.step(3)
        g.step_eager(2)
        outs.append((g.state(), g.residual(), g.info()["fp64_dynamic"]))
        g.close()
    assert np.isfinite(outs[0][0]).all()
    for st, res, dyn in outs[1:]:
        assert np.array_equal(outs[0][0], st)
        assert np.array_equal(outs[0][1], res) and outs[0][2] == dyn


@pytest.mark.parametrize("make,lanes", [SMALL[0], SMALL[5], SMALL[9], SMALL[13]])
def test_cluster_sweeps_match_the_oracle(P, make, lanes):
    sc = make()
    ref = O.OracleScene(sc)
    ref.step(4)
    g = P.Scene(sc, sweep_mode=2, sweep_lanes=lanes)
    for _ in range(3):
        a, b = teacher_forced_step(g, ref)
        assert rel_err(a, b, np.asarray(sc.bodies["he"])) < REL_TOL
    g.close()


@pytest.mark.parametrize("extra", [0, 20000, 70000])
def test_heavy_slices_rank_alike_among_many_bonds(P, extra):
    """Two slabs (about 400 and thousands of bond ends) step bit for bit alike alone and beside
    `extra` boxes on the ground in a group of their own, whose contacts spread the slabs' end ids
    over one, several and more than four windows of the ranking bitmap (and so over its sort)."""
    parts = [S.slab_pile(10), S.slab_pile(40)]
    n_slabs = sum(p.n_bodies for p in parts)
    b = S._bodies(extra)
    k = np.arange(extra)
    b["he"], b["mass"] = 0.5, 1.0
    b["c"] = np.stack([3.0 * (k % 300), np.full(extra, 0.5005), 3.0 * (k // 300)], 1)
    par = dict(parts[0].params, n_iter=3)
    outs = []
    for order in ("slabs first", "boxes first"):
        bodies = [parts[0].bodies.copy(), parts[1].bodies.copy()]
        if extra:
            bodies.insert(0 if order == "boxes first" else 2, b.copy())
        for g, x in enumerate(bodies):
            x["group"] = g
        at = extra if order == "boxes first" else 0
        for mode in (1, 2):
            g = P.Scene(S.Scene("slabs", par, np.concatenate(bodies), S._bonds(0), 1), sweep_mode=mode, sweep_lanes=1)
            g.step(8)
            outs.append(g.state()[at:at + n_slabs])
            if extra and order == "boxes first":
                assert g.info()["n_bonds"] > 4 * extra
            g.close()
    alone = [x.copy() for x in (parts[0].bodies, parts[1].bodies)]
    alone[1]["group"] = 1
    g = P.Scene(S.Scene("slabs", par, np.concatenate(alone), S._bonds(0), 1), sweep_mode=2, sweep_lanes=1)
    g.step(8)
    ref = g.state()
    assert g.info()["heavy_bodies"] == 2
    g.close()
    for o in outs:
        assert np.array_equal(o, ref)


def test_bins_larger_than_shared_memory_are_left_out(P):
    """A group whose iterates do not fit a block's shared memory sweeps as launches."""
    outs = []
    for mode in (2, 1):
        g = P.Scene(_pile(3000), sweep_mode=mode, sweep_lanes=1)
        g.step(2)
        outs.append(g.state())
        g.close()
    assert np.isfinite(outs[0]).all() and np.array_equal(outs[0], outs[1])


def test_step_recaptured_after_a_smaller_scene(P):
    """A scene's step is captured again (for profiling) after a smaller scene with the same sweep
    kernel was set up: its shared memory is still granted."""
    outs = []
    for other in (False, True):
        g = P.Scene(_pile(1024), sweep_mode=2, sweep_lanes=4)
        g.step(1)
        if other:
            h = P.Scene(_groups([5, 9]), sweep_mode=2, sweep_lanes=4)
            h.step(1)
            h.close()
            g.set_profiling(True)
        g.step(2)
        outs.append(g.state())
        g.close()
    assert np.isfinite(outs[0]).all() and np.array_equal(outs[0], outs[1])
