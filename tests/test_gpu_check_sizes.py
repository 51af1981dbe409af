"""Collision verdicts and sphere centres do not depend on how many states a call has: few states run a warp
each, many a lane each with queues between their stages.  Bitwise the same, for every kind of joint, link,
obstacle and pair table the two ways treat differently."""
import dataclasses

import numpy as np
import pytest

from paper_2503_06757_gb300 import prrtc as P
from paper_2503_06757_gb300 import workload as W
from tests import helpers as H

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2503_06757_gb300 import build
    build.build()


def some_pairs(robot, keep):
    """The robot with part of its pairs: link pairs that are no full cross product."""
    pairs = robot.self_pairs[np.random.default_rng(3).random(len(robot.self_pairs)) < keep]
    return dataclasses.replace(robot, self_pairs=pairs)


def turned_boxes(n, seed):
    rng = np.random.default_rng(seed)
    boxes = []
    for _ in range(n):
        q, _ = np.linalg.qr(rng.normal(size=(3, 3)))
        q *= np.sign(np.linalg.det(q))
        a = rng.uniform(0, 2 * np.pi)  # clear of the base
        c = [rng.uniform(0.4, 0.8) * np.cos(a), rng.uniform(0.4, 0.8) * np.sin(a), rng.uniform(0.1, 1.2)]
        boxes.append(np.concatenate([c, rng.uniform(0.02, 0.1, 3), q.reshape(9)]))
    return H.scene(boxes=np.asarray(boxes).astype(np.float32))


def lone_spheres():
    """Links of one sphere, of none and of forty (more than a warp), joints of every type."""
    spheres = [(0, (0.0, 0.0, 0.1), 0.05), (2, (0.05, 0.0, 0.0), 0.04)]
    spheres += [(4, (0.01 * (i % 5), 0.02 * (i // 5), -0.01 * i), 0.03) for i in range(40)]
    pairs = [(0, 1)] + [(0, 2 + i) for i in range(40)] + [(1, 2 + i) for i in range(0, 40, 3)]
    return H.robot([W.JOINT_REV_Z, W.JOINT_PRISM_X, W.JOINT_REV_X, W.JOINT_PRISM_Z, W.JOINT_REV_Y],
                   [0.3, 0.1, 0.2, 0.0, 0.1], lower=[-6.0, -0.3, -3.0, -0.2, -4.0], upper=[6.0, 0.3, 3.0, 0.2, 4.0],
                   spheres=spheres, pairs=pairs)


SETS = {
    "arm7 shelf": lambda: (W.arm7(), W.scene_shelf(1003), {}),
    "arm8 mixed 33": lambda: (W.arm8(), W.scene_mixed(7, 33), {}),
    "dual14 mixed 600": lambda: (W.dual14(), W.scene_mixed(9, 600, bases=W.robot_bases(W.dual14())), {}),
    "dual14 part of the pairs": lambda: (some_pairs(W.dual14(), 0.6), W.scene_shelf(1004, "y"), {}),
    "one box": lambda: (W.arm7(), H.scene(boxes=[H.aabb([0.4, 0.0, 0.6], [0.1, 0.1, 0.1])]), {}),
    "turned boxes": lambda: (W.arm7(), turned_boxes(20, 2), {}),
    "far obstacle": lambda: (W.arm7(), H.scene(spheres=[[40.0, 0.0, 0.0, 1.0]]), {}),
    "empty": lambda: (W.dual14(), H.empty_scene(), {}),
    "no pairs": lambda: (H.no_self(W.arm8()), W.scene_mixed(8, 80), {}),
    "lone spheres": lambda: (lone_spheres(), W.scene_mixed(11, 60), {}),
    "one stage": lambda: (W.arm7(), W.scene_shelf(1005), dict(two_stage=False)),
    "distance field": lambda: (W.arm7(), W.scene_shelf(1006), dict(esdf=True)),
}


@pytest.mark.parametrize("name", list(SETS))
def test_few_and_many_states_agree(name):
    robot, scene, opt = SETS[name]()
    rb, ev = P.make_robot(robot), P.make_env(scene)
    if opt.get("two_stage") is False:
        rb.set_two_stage(False)
    if opt.get("esdf"):
        ev = P.Env.from_occupancy(ev.voxelize((-0.8, -0.8, 0.0), 0.05, (32, 32, 32)), (-0.8, -0.8, 0.0), 0.05)
    n = 6529  # above the limit, no whole warp at the end
    Q = np.random.default_rng(1).uniform(robot.lower, robot.upper, (n, robot.dof)).astype(np.float32)
    valid, spheres = P.prrtc_check_states(rb, ev, Q, want_spheres=True)
    assert 0 < valid.sum() or "600" in name
    plain = P.prrtc_check_states(rb, ev, Q)  # without centres
    np.testing.assert_array_equal(plain, valid)
    # up to 1024 states go through pinned host memory, unless their centres are too many
    for lo, hi in ((0, 1), (1, 34), (34, 1058), (1058, 2083), (2083, n)):
        np.testing.assert_array_equal(P.prrtc_check_states(rb, ev, Q[lo:hi]), valid[lo:hi])
        assert P.prrtc_last_launch_stats()["fk_states"] == hi - lo
        v, s = P.prrtc_check_states(rb, ev, Q[lo:hi], want_spheres=True)
        np.testing.assert_array_equal(v, valid[lo:hi])
        np.testing.assert_array_equal(s, spheres[lo:hi])
