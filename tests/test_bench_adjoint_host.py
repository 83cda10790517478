"""bench.py's account of the adjoint: launches of the reverse, counted in the
source of the function that queues them, and groups that are timed.  No GPU is
needed."""
import importlib.util
import os
import re

import paper_1806_10550_gb300 as tf

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
_spec = importlib.util.spec_from_file_location("bench_under_test", os.path.join(ROOT, "bench.py"))
bench = importlib.util.module_from_spec(_spec)
_spec.loader.exec_module(bench)


def launches(code):
    return len(re.findall(r"<<<|ops->solve_t\(", code))


def test_reverse_launches_are_those_of_the_source():
    with open(os.path.join(bench.CSRC, "tf_adjoint.cu")) as f:
        src = f.read()
    body = src[src.index("int adj_reverse("):]
    body = body[:body.index("\n}")]
    loop = body[body.index("for (int k = K - 1; k >= 0; --k) {"):]
    loop = loop[:loop.index("\n  }")]
    per_iteration, per_step = launches(loop), launches(body) - launches(loop)
    assert per_iteration > 0 and per_step > 0
    for K, ns in ((1, 1), (3, 400), (5, 7)):
        groups, total = bench.adjoint_reverse_launches(K, ns)
        assert total == ns * (per_iteration * K + per_step)
        assert groups["solve_t"] == ns * K * len(re.findall(r"ops->solve_t\(", loop))
        assert groups["line_x"] == ns * K * loop.count("k_vjp_iter<<<")
        assert groups["D"] == ns * (body.count("k_vjp_D<<<") - loop.count("k_vjp_D<<<"))


def test_every_accounted_group_is_timed():
    groups, _ = bench.adjoint_reverse_launches(3, 2)
    assert set(groups) == set(bench.ADJ_BYTES_PER_CELL)
    assert set(groups) <= set(tf.ADJOINT_GROUPS)
    with open(os.path.join(bench.CSRC, "tf_adjoint.cu")) as f:
        src = f.read()
    timed = dict(zip(("kGForward", "kGBand", "kGSolve", "kGLineX", "kGLineY", "kGD", "kGKappa"), tf.ADJOINT_GROUPS))
    used = {timed[g] for g in re.findall(r"T\.begin\((kG\w+)\)", src)}
    assert set(groups) <= used
