"""The near-root kernel of the per-level forms, and small games resident in
one CTA (the default form's choice): bitwise the oracle in FP64, whatever the
depth at which the launches take over, rule, order, or split of the calls."""
import numpy as np
import pytest
import torch

import gamegen as gg
import oracle
from paper_2609_11923_gb300 import cfr

from tests.fp32_band import fp32_band, fp32_bar
from tests.test_gpu_batch import chain_game
from tests.test_gpu_set_edges import two_level_game

pytestmark = pytest.mark.gpu

GAMES = [("tree%d" % d, lambda d=d: gg.random_tree(11, depth=d)) for d in (3, 4, 5, 7, 9, 11)] + [
    ("leduc", gg.leduc), ("kuhn", gg.kuhn), ("endgame", lambda: gg.endgame(2, 30000)),
    ("card", lambda: gg.large_card(3, 2, 2, 3)), ("chain40", lambda: chain_game(40)),
    ("sets", lambda: two_level_game(300, 8, 7)), ("one_action", lambda: two_level_game(9, 1, 1))]
FORMS = {"auto": cfr.EXEC_AUTO, "graph": cfr.EXEC_GRAPH, "levels": cfr.EXEC_LEVELS}


@pytest.mark.parametrize("name,make", GAMES)
@pytest.mark.parametrize("form", list(FORMS))
def test_fp64_equals_the_oracle(form, name, make):
    g = make()
    for rule, orule, order in ((cfr.RULE_CFR_PLUS, oracle.CFR_PLUS, 0), (cfr.RULE_PCFR_PLUS, oracle.PCFR_PLUS, 1),
                               (cfr.RULE_CFR, oracle.CFR, 0)):
        s = cfr.Solver(g, precision=cfr.P64, exec_form=FORMS[form], rule=rule, order=order)
        for n in (1, 6, 13):  # a call goes on where the one before ended
            s.iterate(n)
        s.synchronize()
        R, avg, t = s.get_state()
        o = oracle.solve(g, 20, rule=orule, order=order)
        assert t == 20
        np.testing.assert_array_equal(R, o.R)
        np.testing.assert_array_equal(avg, o.sbar)
        s.close()


@pytest.mark.parametrize("overlap", [cfr.OVERLAP_ON, cfr.OVERLAP_OFF])
@pytest.mark.parametrize("order", [0, 1])
def test_overlap_graph_length_and_profile_leave_the_same_bits(order, overlap):
    g = gg.random_tree(3, depth=10)
    ref = cfr.Solver(g, precision=cfr.P32, exec_form=cfr.EXEC_LEVELS, order=order, launch_overlap=cfr.OVERLAP_OFF)
    ref.iterate(23)
    s = cfr.Solver(g, precision=cfr.P32, exec_form=cfr.EXEC_GRAPH, order=order, launch_overlap=overlap, graph_iters=7)
    s.iterate(9)
    s.iterate(14)
    for a, b in zip(s.get_state(), ref.get_state()):
        np.testing.assert_array_equal(a, b)


def test_fp32_resident_games_reach_the_oracle_exploitability():
    # bar: 1e-4 of the pot, or what payoffs perturbed by FP32's unit roundoff
    # move the oracle itself by (fp32_band; Leduc is such a case)
    for make in (gg.tiny_card, gg.leduc, lambda: gg.random_tree(4, depth=8), lambda: gg.endgame(9, 6000)):
        g = make()
        s = cfr.Solver(g, precision=cfr.P32)
        s.iterate(1000)
        want, delta = fp32_band(make, 1000)
        assert abs(s.exploitability() - want) <= fp32_bar(g.pot, delta)
        s.reset()
        s.iterate(1000)  # runs repeat
        a = s.get_state()
        s.reset()
        s.iterate(400)
        s.iterate(600)
        for x, y in zip(a, s.get_state()):
            np.testing.assert_array_equal(x, y)
        s.close()
