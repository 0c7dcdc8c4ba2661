"""The one-launch front of small scenes finds the same pairs and contacts as the kernels for larger
ones (which pabd_detect runs) and the oracle, at the sizes where it starts and stops and where its
lists outgrow shared memory, and steps as the oracle does."""
import numpy as np
import pytest

import oracle as O
import scenes as S
from gpu_helpers import REL_TOL, rel_err, same_contacts, teacher_forced_step

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


def _cloud(n, side, groups=1, bonds=0, contacts=1):
    rng = np.random.default_rng(100 + n)
    b = S._bodies(n)
    b["he"] = rng.uniform(0.1, 0.3, (n, 3))
    b["mass"] = rng.uniform(0.5, 2.0, n)
    b["c"] = rng.uniform(0.0, side, (n, 3))
    b["quat"] = S._random_unit_quats(rng, n)
    b["pinned"][rng.random(n) < 0.2] = 1
    b["group"] = np.arange(n) * groups // n
    bo = S._bonds(bonds)
    for k in range(bonds):
        g = np.nonzero(b["group"] == b["group"][k % n])[0]
        i, j = g[k % len(g)], g[(k + 1) % len(g)]
        bo["type"][k], bo["i"][k], bo["j"][k] = (S.SPHERICAL, S.SPRING)[k % 2], i, j if i != j else S.WORLD
        bo["kappa"][k], bo["rest"][k] = 50.0, 0.2
    return S.Scene("cloud", S.default_params(n_iter=4, body_contacts=contacts), b, bo, 1)


CASES = [(1, 0.5, 1, 0, 1), (2, 0.2, 1, 1, 1), (31, 1.0, 1, 20, 1), (33, 1.2, 4, 10, 1), (64, 1.5, 1, 0, 1),
         (127, 2.5, 3, 60, 1), (128, 2.5, 1, 0, 1), (129, 2.5, 1, 0, 1),
         (60, 0.15, 1, 0, 1),   # more than 1024 pairs, bodies with hundreds of ends
         (1, 0.2, 1, 0, 0), (32, 0.3, 5, 16, 0), (33, 0.3, 5, 16, 0)]


@pytest.mark.parametrize("n,side,groups,bonds,contacts", CASES)
def test_small_front_equals_detection_and_oracle(P, n, side, groups, bonds, contacts):
    sc = _cloud(n, side, groups, bonds, contacts)
    cap = dict(max_pairs=max(64, 40 * n), max_contacts=max(64, 400 * n))
    ref = O.OracleScene(sc)
    st = ref.state()
    outs = []
    for run in ("detect", "step", "step_eager"):
        g = P.Scene(sc, **cap)
        g.set_state(st)
        g.detect() if run == "detect" else getattr(g, run)(1)
        outs.append((g.pairs(), g.contacts(), g.info()["offgrid_bodies"]))
        if run != "detect":
            assert np.isfinite(g.state()).all()
        g.close()
    ref.detect()
    assert np.array_equal(outs[0][0], ref.pairs())
    for pairs, cont, off in outs[1:]:
        assert np.array_equal(pairs, outs[0][0]) and off == outs[0][2]
        assert np.array_equal(cont[0], outs[0][1][0]) and np.array_equal(cont[1], outs[0][1][1])
    same_contacts(outs[1][1], ref.contacts())


def test_small_front_reports_capacity(P):
    g = P.Scene(_cloud(40, 0.3), max_pairs=16, max_contacts=20)
    g.step(1)
    assert g.sync(allow=(P.ERR_CAPACITY,)) == P.ERR_CAPACITY
    i = g.info()
    assert i["n_pairs"] == 16 and i["n_contacts"] <= 20
    g.close()


@pytest.mark.parametrize("make", [lambda: S.chain_pendulum(n_bodies=5), lambda: S.slab_pile(7),
                                  lambda: S.box_pile_n(40, stacked=True)])
def test_small_front_steps_match_the_oracle(P, make):
    sc = make()
    ref = O.OracleScene(sc)
    g = P.Scene(sc)
    for k in range(6):
        a, b = teacher_forced_step(g, ref)
        assert rel_err(a, b, np.asarray(sc.bodies["he"])) < REL_TOL, k
    g.close()
