"""A wait of collision detection that runs out changes nothing: with the bound at one poll the narrow
phase counts late tiles again itself, and pairs, contacts and states are those of the default bound."""
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


# two tiles and no pair, a last tile of one body, tiles of pairs alone, hundreds of tiles, one body
# in thousands of pairs; and lists cut at their capacity (0: the default)
@pytest.mark.parametrize("make,max_contacts", [
    (lambda: S.box_pile_n(129), 0), (lambda: S.box_pile_n(257, stacked=True), 0),
    (lambda: S.box_pile_n(5000, stacked=True, spacing=1.2), 0), (lambda: S.box_pile_n(20011, stacked=True), 0),
    (lambda: S.slab_pile(40), 0), (lambda: S.box_pile_n(5000, stacked=True), 3001),
    (lambda: S.box_pile_n(2000, stacked=True), 1)])
def test_shortest_wait_gives_the_same_contacts_and_states(P, make, max_contacts):
    want = P.OK if max_contacts == 0 else P.ERR_CAPACITY
    outs = []
    for polls in (None, 1):
        for mode in (1, 2):
            g = P.Scene(make(), sweep_mode=mode, max_contacts=max_contacts)
            if polls:
                g.set_wait_limit(polls)
            g.detect()
            assert g.sync(allow=(want,)) == want
            out = [g.pairs(), *g.contacts()]
            if want == P.OK:
                g.step(3)
                g.step_eager(1)
                assert g.sync() == P.OK
                out.append(g.state())
            outs.append(out)
            g.close()
    assert all(np.isfinite(x).all() for x in outs[0])
    for out in outs[1:]:
        assert all(np.array_equal(a, b) for a, b in zip(outs[0], out))
