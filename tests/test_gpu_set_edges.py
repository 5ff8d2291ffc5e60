"""Sets at the edges of the lane groups: one set of M members and A actions
above A sets of M members and B actions, M around the group and block sizes
and actions around the register tiers. FP64 sums run one chain per slot and
must equal the oracle bitwise whatever the group."""
import numpy as np
import pytest
import torch

import gamegen as gg
import oracle
from paper_2609_11923_gb300 import cfr

pytestmark = pytest.mark.gpu


def two_level_game(m, a, b, seed=0):
    """Chance over m outcomes; player 1 (one set, a actions) does not see
    which; player 2 (b actions) sees player 1's action only. Random payoffs."""
    rng = np.random.default_rng(1000 * seed + 100 * m + 10 * a + b)
    p = rng.gamma(1.0, size=m)
    nodes = [(gg.CHANCE, -1, list(range(1, m + 1)), list(p / p.sum()), 0.0)]
    nodes += [None] * m
    for k in range(1, m + 1):
        kids = []
        for i in range(a):
            leaves = []
            for _ in range(b):
                leaves.append(len(nodes))
                nodes.append((gg.TERMINAL, -1, [], None, float(rng.uniform(-1, 1))))
            kids.append(len(nodes))
            nodes.append((gg.P2, 1 + i, leaves, None, 0.0))
        nodes[k] = (gg.P1, 0, kids, None, 0.0)
    return gg.from_lists(nodes, [(0, a)] + [(1, b)] * a)


@pytest.mark.parametrize("lanes", [1, 2, 4, 8, 16, 32, 256])
@pytest.mark.parametrize("a,b", [(2, 3), (4, 4), (5, 2), (8, 7)])
def test_fp64_sums_equal_the_oracle_at_every_group_edge(lanes, a, b):
    for m in (1, 3, 4, 7, 8, 9, 16, 17, 31, 33, 255, 257):
        g = two_level_game(m, a, b)
        s = cfr.Solver(g, precision=cfr.P64, exec_form=cfr.EXEC_LEVELS, lanes_per_set=lanes)
        s.iterate(30)
        R, avg, _ = s.get_state()
        o = oracle.solve(g, 30)
        np.testing.assert_array_equal(R, o.R, err_msg="m=%d" % m)
        np.testing.assert_array_equal(avg, o.sbar, err_msg="m=%d" % m)
        s.close()


@pytest.mark.parametrize("a,b", [(2, 3), (3, 2), (4, 1), (5, 8)])
@pytest.mark.parametrize("m", [1, 31, 32, 33, 63, 65, 170, 257, 800])
def test_streamed_sets_at_the_edges_of_teams_and_steps(m, a, b):
    """One set of the streaming backward, from one member to stages so large
    that few teams fit. One iteration from the uniform strategy: a regret is a
    sum of m terms that add up to at most 2 in size (payoffs in [-1, 1] times
    the deal's probabilities), each with a few roundings, in sums of at most
    m / 32 + 12 terms one after another."""
    g = two_level_game(m, a, b)
    s = cfr.Solver(g, precision=cfr.P32, exec_form=cfr.EXEC_LEVELS, lanes_per_set=cfr.STREAM_LANES)
    assert cfr.cfr_export_array(s.h, "stream_ok")[1:].all()
    s.iterate(1)
    s.synchronize()
    R, avg, _ = s.get_state()
    o = oracle.solve(g, 1)
    tol = 2.0 * (m / 32 + 12 + 12) * 2.0 ** -24
    assert np.abs(R - o.R).max() <= tol
    assert (np.abs(avg - o.sbar) <= tol * o.sbar).all()
    s.close()


def mixed_sets_game(most):
    """One depth of player 1's and player 2's sets of 1 to 70 members and 2 to
    `most` actions, side by side in the same warps; random payoffs."""
    rng = np.random.default_rng(most)
    sets = [(m, 2 + (i * 5 + m) % (most - 1)) for i, m in enumerate([1, 2, 5, 9, 33, 3, 70, 4, 8, 17, 1, 31, 32, 6] * 3)]
    members = [I for I, (m, _) in enumerate(sets) for _ in range(m)]
    p = rng.gamma(1.0, size=len(members))
    nodes = [(gg.CHANCE, -1, list(range(1, len(members) + 1)), list(p / p.sum()), 0.0)] + [None] * len(members)
    for k, I in enumerate(members):
        leaves = []
        for _ in range(sets[I][1]):
            leaves.append(len(nodes))
            nodes.append((gg.TERMINAL, -1, [], None, float(rng.uniform(-1, 1))))
        nodes[1 + k] = (gg.P1 if I % 3 else gg.P2, I, leaves, None, 0.0)
    return gg.from_lists(nodes, [(0 if I % 3 else 1, a) for I, (_, a) in enumerate(sets)])


@pytest.mark.parametrize("order", [cfr.ORDER_SIMULTANEOUS, cfr.ORDER_ALTERNATING])
@pytest.mark.parametrize("lanes", [0, 4, 8, 16, 32])
@pytest.mark.parametrize("most", [4, 8])
def test_sets_of_different_sizes_share_a_warp(most, lanes, order):
    g = mixed_sets_game(most)
    s = cfr.Solver(g, precision=cfr.P64, exec_form=cfr.EXEC_LEVELS, lanes_per_set=lanes, order=order)
    s.iterate(30)
    R, avg, _ = s.get_state()
    o = oracle.solve(g, 30, order=order)
    np.testing.assert_array_equal(R, o.R)
    np.testing.assert_array_equal(avg, o.sbar)
    s.close()


def seconds(s, n=20):
    s.iterate(n)
    torch.cuda.synchronize()
    best = 1e9
    for _ in range(5):
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record()
        s.iterate(n)
        e1.record()
        torch.cuda.synchronize()
        best = min(best, e0.elapsed_time(e1))
    return best


def test_short_sets_do_not_pay_for_the_lanes_of_a_group():
    # sets of one member by groups of 32 lanes: no slower than by groups of 4
    from tests.test_gpu_batch import chain_game

    took = {}
    for lanes in (4, 32):
        s = cfr.Solver(chain_game(40), precision=cfr.P64, exec_form=cfr.EXEC_PERSISTENT, lanes_per_set=lanes)
        took[lanes] = seconds(s)
        s.close()
    assert took[32] < 1.12 * took[4], took


@pytest.mark.parametrize("g", [two_level_game(300, 5, 8), two_level_game(1000, 2, 2), gg.random_tree(1, depth=8)],
                         ids=["300x5x8", "1000x2x2", "rt8"])
def test_tuning_is_not_slower_than_a_shape_that_it_tries(g):
    # long sets near the root, and a game at the edge of the resident form
    fixed = []
    for lanes in (8, 32, 256):
        s = cfr.Solver(g, precision=cfr.P64, exec_form=cfr.EXEC_GRAPH, lanes_per_set=lanes)
        fixed.append(seconds(s))
        s.close()
    s = cfr.Solver(g, precision=cfr.P64)
    s.autotune()
    tuned = seconds(s)
    s.reset()
    s.iterate(9)
    np.testing.assert_array_equal(s.avg_strategy(), oracle.solve(g, 9).avg_strategy())
    s.close()
    assert tuned < 1.35 * min(fixed), (tuned, fixed)  # 1.0 measured, 1.5 to 2.5 with the forms untried
