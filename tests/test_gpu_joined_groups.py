"""User bonds between bodies of different groups: the groups share no contacts but step together, the
same bit for bit in every sweep mode and as the oracle has it."""
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


def _chain(n, per, step):
    """The chain pendulum with `per` bodies to a group, and springs that reach `step` bodies along."""
    sc = S.chain_pendulum(n_bodies=n)
    sc.bodies["group"] = np.arange(n) // per
    far = S._bonds(len(range(0, n - step, 7)) if step else 0)
    for k, i in enumerate(range(0, n - step, 7) if step else ()):
        far[k]["type"], far[k]["i"], far[k]["j"] = S.SPRING, i + step, i
        far[k]["kappa"], far[k]["rest"] = 50.0, np.linalg.norm(sc.bodies["c"][i] - sc.bodies["c"][i + step])
    sc.bonds = np.concatenate([sc.bonds, far])
    return sc


# joints between neighbouring groups of a block's size, of one body, uneven, and springs across the
# whole scene; and groups of one bin each, joined by nothing (the sweeps then need one launch)
@pytest.mark.parametrize("n,per,step,apart", [(16, 8, 0, False), (12, 1, 0, False), (300, 9, 0, False),
                                              (300, 40, 250, False), (40, 40, 30, True)])
def test_bonds_between_groups(P, n, per, step, apart):
    outs = []
    for mode, order in ((2, 1), (1, 1), (3, 0), (0, 0)):
        g = P.Scene(_chain(n, per, step), sweep_mode=mode, light_order=order)
        g.set_profiling(True)
        g.step(2)
        p = g.profile()
        if mode == 2:
            assert p["sweep_launches"] == (p["steps"] if apart else p["sweeps"])
        g.set_profiling(False)
        g.step(2)
        g.step_eager(1)
        outs.append(np.concatenate([g.state().ravel(), g.residual()]))
        g.close()
    assert np.isfinite(outs[0]).all()
    assert all(np.array_equal(outs[0], o) for o in outs[1:])
    sc = _chain(n, per, step)
    ref = O.OracleScene(sc)
    g = P.Scene(sc, sweep_mode=2, light_order=1)
    for _ in range(3):
        a, b = teacher_forced_step(g, ref)
        assert rel_err(a, b, sc.bodies["he"]) < REL_TOL
    g.close()
