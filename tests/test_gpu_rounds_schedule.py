"""How many rounds of a serial or lockstep plan run side by side, and on how many blocks, follows from what its
rounds have changed lately and from how many problems are still open.  The plans and their counters do not:
batches in which a few problems without a solution outlast many easy ones (so that they go through all launches),
in which nearly every round changes a tree or a radius, and which end within their first round, against one
round at a time."""
import numpy as np
import pytest

from paper_2503_06757_gb300 import prrtc as P
from paper_2503_06757_gb300 import workload as W
from tests import helpers as H
from tests.test_gpu_rounds import problems, same, shelf

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2503_06757_gb300 import build
    build.build()


def rooms(n, closed):
    """n problems of the point robot, every one through the door of its own kind: `closed` of them shut."""
    rb = P.make_robot(H.point_robot())
    wide = P.make_env(W.scene_two_rooms(door=(0.4, 0.8)))
    shut = P.make_env(H.scene(boxes=[H.aabb([0.6, 0.0, 0.5], [0.01, 2.0, 2.0])]))
    s, g = W.two_rooms_pairs(n, 3)
    return [(rb, shut if k % (n // closed) == 1 else wide, s[k], g[k], 5 + k, 0) for k in range(n)]


POINT = dict(range=0.2, resolution=0.01, tree_capacity=4096, path_capacity=4096)
CASES = {
    "easy and closed": (lambda: rooms(200, 4), dict(POINT, max_iters=2500)),
    "many closed": (lambda: rooms(160, 60), dict(POINT, max_iters=1400)),
    "few, closed": (lambda: rooms(5, 2), dict(POINT, max_iters=1400)),
    "radii": (lambda: problems(W.arm7(), shelf(W.arm7(), 4), 160),
              dict(max_iters=300, dd_radius=5.0, dd_alpha=0.02, dd_min_radius=4.0)),
    "one round": (lambda: problems(W.arm7(), shelf(W.arm7(), 4), 200), dict(max_iters=5)),
}


@pytest.mark.parametrize("name", list(CASES))
def test_serial(name):
    make, kw = CASES[name]
    items = make()
    prm = P.params(mode=P.MODE_SERIAL, **dict(dict(tree_capacity=4096, path_capacity=4096), **kw))
    got = P.prrtc_plan_batch(items, prm)
    if "closed" in name:
        assert any(r["iterations"] == kw["max_iters"] for r in got) and any(r["status"] == P.SOLVED for r in got)
    for k in list(range(0, len(items), 7)) + [k for k, r in enumerate(got) if r["status"] != P.SOLVED][:6]:
        prm.seed = items[k][4]
        same(got[k], P.prrtc_plan_noalloc(*items[k][:4], prm), (name, k))


@pytest.mark.parametrize("workers", [2, 8, 33])
@pytest.mark.parametrize("name", list(CASES))
def test_lockstep(name, workers):
    make, kw = CASES[name]
    items = make()
    kw = dict(dict(mode=P.MODE_LOCKSTEP, workers=workers, tree_capacity=4096, path_capacity=4096), **kw)
    want = P.prrtc_plan_batch(items, P.params(warps_per_block=min(workers, 4), **kw))
    got = P.prrtc_plan_batch(items, P.params(**kw))
    for k in range(len(items)):
        same(got[k], want[k], (name, workers, k))


def test_tuner_leaves_the_tile_of_serial_plans_alone():
    """Serial rounds have one obstacle tile: the tuner does not choose between two."""
    items = problems(W.arm7(), shelf(W.arm7(), 2), 4)
    prm = P.params(mode=P.MODE_SERIAL, max_iters=50, tree_capacity=4096)
    assert all(P.prrtc_autotune(items, prm, trials=1)[0].obstacle_tile == 32 for _ in range(12))
