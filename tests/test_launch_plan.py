"""What cfr_iterate launches, by the options (host only)."""
import pytest

import gamegen as gg
from paper_2609_11923_gb300 import cfr


def plan(g, **kw):
    h = cfr.cfr_compile(g, cfr.make_options(**kw))
    try:
        return cfr.cfr_launch_plan(h)
    finally:
        cfr.cfr_destroy(h)


@pytest.mark.parametrize("precision", [cfr.P32, cfr.P64])
@pytest.mark.parametrize("kw", [{}, {"graph_iters": 10}, {"launch_overlap": cfr.OVERLAP_OFF},
                                {"launch_overlap": cfr.OVERLAP_ON, "graph_iters": 3}])
def test_options_that_leave_the_results_alone_do_not_choose_the_form(precision, kw):
    # the resident form's FP32 sums have last bits of their own
    assert plan(gg.tiny_card(), precision=precision, **kw)["resident_threads"] > 0
    assert plan(gg.random_tree(3, depth=10), precision=precision, **kw)["near_root_depth"] > 0


@pytest.mark.parametrize("kw", [{"exec_form": cfr.EXEC_GRAPH}, {"exec_form": cfr.EXEC_LEVELS}, {"exec_form": cfr.EXEC_PERSISTENT},
                                {"lanes_per_set": 8}, {"persistent_ctas": 2}, {"reach_order": cfr.REACH_BFS}])
def test_a_form_or_a_shape_that_is_asked_for_is_the_one_that_runs(kw):
    p = plan(gg.tiny_card(), **kw)
    assert p["resident_threads"] == 0
    if "lanes_per_set" in kw or "reach_order" in kw:
        assert p["near_root_depth"] == -1


def test_launches_overlap_where_the_option_says():
    g, off, on = gg.tiny_card(), cfr.OVERLAP_OFF, cfr.OVERLAP_ON
    for precision in (cfr.P32, cfr.P64):
        for overlap, want in ((off, (0, 0)), (on, (1, 1)), (cfr.OVERLAP_AUTO, (1, 1))):
            p = plan(g, precision=precision, launch_overlap=overlap)
            assert (p["overlap"], p["evaluation_overlap"]) == want
    p = plan(gg.random_tree(3, depth=11), precision=cfr.P64)  # more than 100,000 nodes
    assert (p["overlap"], p["evaluation_overlap"]) == (0, 1)


def test_the_resident_line_lies_where_the_forms_cross():
    # FP64: 3,385 nodes 52.6 us resident and 38.5 as a graph, 2,341 nodes 18.1 and 24.8
    assert plan(gg.random_tree(1, depth=8), precision=cfr.P64)["resident_threads"] == 0
    assert plan(gg.tiny_card(13, 2), precision=cfr.P64)["resident_threads"] > 0
    assert plan(gg.random_tree(1, depth=8), precision=cfr.P32)["resident_threads"] > 0
