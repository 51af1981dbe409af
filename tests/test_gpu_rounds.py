"""Serial and lockstep plans run several rounds side by side and keep those that
count: bitwise the plans, and the counters, of one round at a time.

Serial batches are compared with prrtc_plan_noalloc, which runs one warp in the
order of Alg. 1; lockstep batches with a launch whose warps per block are given,
which runs one round at a time on one block.  Batch sizes 1 .. 170 take every
sequence of launches (clusters of 16, 8 .. 1 blocks first, then larger ones)."""
import numpy as np
import pytest

from paper_2503_06757_gb300 import learned as L
from paper_2503_06757_gb300 import prrtc as P
from paper_2503_06757_gb300 import workload as W
from tests import helpers as H

pytestmark = pytest.mark.gpu

SCALARS = ("status", "n", "iterations", "cost", "nodes_a", "nodes_b", "edges_checked", "edge_states", "sphere_tests",
           "pair_tests", "fk_states", "nn_nodes", "dd_rejected", "prim_tests", "verdict_states")


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2503_06757_gb300 import build
    build.build()


def same(a, b, what, names=SCALARS):
    for name in names:
        assert a[name] == b[name], (what, name, a[name], b[name])
    np.testing.assert_array_equal(a["path"], b["path"])


def problems(robot, scenes, n, esdf=False):
    """n free pairs over the scenes, the goals inside a cubby."""
    rb, out = P.make_robot(robot), []
    envs = [P.make_env(sc) for sc in scenes]
    pairs = [(k, *pair) for k, (sc, ev) in enumerate(zip(scenes, envs))
             for pair in zip(*L.scene_pairs(robot, sc, rb, ev, 20, 50 + k, chunk=4096))]
    assert pairs
    if esdf:
        envs = [P.Env.from_occupancy(ev.voxelize((-0.8, -0.8, 0.0), 0.05, (32, 32, 32)), (-0.8, -0.8, 0.0), 0.05)
                for ev in envs]
    for i in range(n):
        k, start, goal = pairs[i * 7 % len(pairs)]
        out.append((rb, envs[k], start, goal, 3 + i, 0))
    return out


def shelf(robot, n):
    return [W.scene_shelf(1000 + k, W.shelf_facing(robot)) for k in range(n)]


CASES = {
    "plain": (lambda: problems(W.arm7(), shelf(W.arm7(), 6), 6), dict(max_iters=3000)),
    "one": (lambda: problems(W.arm7(), shelf(W.arm7(), 1), 1), dict(max_iters=3000)),
    "wave of 4": (lambda: problems(W.arm7(), shelf(W.arm7(), 8), 30), dict(max_iters=1500)),
    "three launches": (lambda: problems(W.arm7(), shelf(W.arm7(), 10), 170), dict(max_iters=1301)),
    "two arms": (lambda: problems(W.dual14(), shelf(W.dual14(), 3), 5), dict(max_iters=700)),
    "halton": (lambda: problems(W.arm7(), shelf(W.arm7(), 3), 3), dict(max_iters=900, sampler=P.SAMPLER_HALTON)),
    "dynamic domain": (lambda: problems(W.arm7(), shelf(W.arm7(), 4), 4),
                       dict(max_iters=900, dd_radius=5.0, dd_alpha=0.1, dd_min_radius=1.0)),
    "distance field": (lambda: problems(W.arm7(), shelf(W.arm7(), 3), 4, esdf=True), dict(max_iters=600)),
    "full trees": (lambda: problems(W.arm7(), shelf(W.arm7(), 4), 4), dict(max_iters=900, tree_capacity=6)),
    "short edges": (lambda: problems(W.arm7(), shelf(W.arm7(), 4), 4), dict(max_iters=37, range=0.06)),
    # held rows above their limit: one warp a problem, as without rounds
    "tiny range": (lambda: problems(W.dual14(), shelf(W.dual14(), 2), 70), dict(max_iters=5, range=0.005)),
}


@pytest.mark.parametrize("name", list(CASES))
def test_serial_rounds_equal_one_warp(name):
    make, kw = CASES[name]
    items = make()
    prm = P.params(mode=P.MODE_SERIAL, **dict(dict(tree_capacity=4096, path_capacity=4096), **kw))
    got = P.prrtc_plan_batch(items, prm)
    for k, it in enumerate(items):
        prm.seed = it[4]
        want = P.prrtc_plan_noalloc(*it[:4], prm)
        same(got[k], want, (name, k))
    if name == "three launches":
        assert P.prrtc_last_launch_stats()["problems"] == 170
        assert max(r["iterations"] for r in got) > 1024  # the third launch had work


@pytest.mark.parametrize("workers", [1, 3, 8, 40, 300])
@pytest.mark.parametrize("name", ["one", "plain", "dynamic domain", "full trees", "three launches"])
def test_lockstep_rounds_equal_one_at_a_time(name, workers):
    make, kw = CASES[name]
    items = make()[:48 if workers > 8 else None]
    kw = dict(dict(mode=P.MODE_LOCKSTEP, workers=workers, tree_capacity=4096, path_capacity=4096), **kw)
    want = P.prrtc_plan_batch(items, P.params(warps_per_block=min(workers, 3), **kw))
    got = P.prrtc_plan_batch(items, P.params(**kw))
    for k in range(len(items)):
        same(got[k], want[k], (name, workers, k))


def test_lockstep_mixture_and_time_limit():
    """A mixture is drawn from by the iteration's own words; a spent time limit ends the problem."""
    robot = W.arm7()
    items = [it + (W.random_mixture(robot.dof, 5).astype(np.float32),) for it in problems(robot, shelf(robot, 2), 4)]
    kw = dict(mode=P.MODE_LOCKSTEP, workers=4, learned_ratio=0.5, max_iters=500, tree_capacity=4096)
    want = P.prrtc_plan_batch(items, P.params(warps_per_block=4, **kw))
    got = P.prrtc_plan_batch(items, P.params(**kw))
    for k in range(len(items)):
        same(got[k], want[k], k)
    walled = H.scene(boxes=[H.aabb([0.6, 0.0, 0.5], [0.01, 2.0, 2.0])])  # no way through
    rb, ev = P.make_robot(H.point_robot()), P.make_env(walled)
    r = P.prrtc_plan(rb, ev, [0.1, 0.1], [1.1, 0.1], P.params(mode=P.MODE_SERIAL, max_iters=1 << 30,
                                                             tree_capacity=1 << 14, time_limit_s=0.05))
    assert r["status"] == P.TIME_LIMIT
