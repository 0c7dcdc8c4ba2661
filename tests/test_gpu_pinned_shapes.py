"""The sweep's launch shapes with nothing left to the tuner's timing: with sweep_mode and light_order both
given, the groups that fit clusters take the one launch for all sweeps, and the lanes' threads are
halved from the size on where they would not all be resident.  Every shape computes the compared
states here, and they are the same bit for bit."""
import numpy as np
import pytest

import oracle as O
import scenes as S
from gpu_helpers import REL_TOL, rel_err, teacher_forced_step
from test_gpu_sweep_shapes import SMALL, _pile

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


def _resident():
    """Threads of the sweep kernels that the device holds at once."""
    import torch
    return torch.cuda.get_device_properties(0).multi_processor_count * 4 * 128


def _run(P, sc, mode, lanes):
    """(sweep launches per step, state, residual, redone bodies) after a few steps."""
    g = P.Scene(sc, sweep_mode=mode, sweep_lanes=lanes, light_order=1)
    assert g.info()["tuned"] == 0
    g.set_profiling(True)
    g.step(2)
    p = g.profile()
    g.set_profiling(False)
    g.step(1)
    g.step_eager(2)
    out = g.state(), g.residual(), g.info()["fp64_dynamic"]
    g.close()
    assert np.isfinite(out[0]).all()
    return p["sweep_launches"] / p["steps"], p["sweeps"] / p["steps"], out


def _same(a, b):
    return all(np.array_equal(x, y) for x, y in zip(a, b))


# (of SMALL, the scenes whose groups all fit clusters: a body too many and 12 clusters of 16 blocks do not)
@pytest.mark.parametrize("k", [k for k in range(len(SMALL)) if k not in (2, 6)])
def test_clusters(P, k):
    make, lanes = SMALL[k]
    launches, sweeps, out = _run(P, make(), 2, lanes)
    assert launches == 1
    for mode in (1, 3):
        n, _, other = _run(P, make(), mode, lanes)
        assert n == (2 * sweeps if mode == 1 else 1)
        assert _same(out, other), mode


@pytest.mark.parametrize("lanes", [16, 8, 4, 2])
@pytest.mark.parametrize("past", [0, 1])
def test_a_thread_per_lane_or_per_two(P, lanes, past):
    n = _resident() // lanes + past
    launches, sweeps, out = _run(P, _pile(n), 2, lanes)
    assert launches == sweeps
    for mode in (1, 3):
        assert _same(out, _run(P, _pile(n), mode, lanes)[2]), mode


@pytest.mark.parametrize("make,lanes", [(lambda: _pile(200), 16), (lambda: S.chain_pendulum(n_bodies=30), 16),
                                        (lambda: S.slab_pile(10), 16), (lambda: S.batched_trees(n_scenes=5), 16)])
def test_clusters_match_the_oracle(P, make, lanes):
    sc = make()
    ref = O.OracleScene(sc)
    ref.step(4)
    g = P.Scene(sc, sweep_mode=2, sweep_lanes=lanes, light_order=1)
    g.set_profiling(True)
    for _ in range(3):
        a, b = teacher_forced_step(g, ref)
        assert rel_err(a, b, np.asarray(sc.bodies["he"])) < REL_TOL
    assert g.profile()["sweep_launches"] == 3
    g.close()
