"""Links skip the obstacles when they stay clear of a box around them all: verdicts of many states (which use the
box) are those of few (which do not), for boxes whose rotation is not quite one, and after obstacles have moved."""
import numpy as np
import pytest

from paper_2503_06757_gb300 import prrtc as P
from paper_2503_06757_gb300 import workload as W
from tests import helpers as H
from tests.test_gpu_check_sizes import turned_boxes

pytestmark = pytest.mark.gpu

N = 6529  # above the limit up to which a state has a warp


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2503_06757_gb300 import build
    build.build()


def box(c, h, rows):
    return np.concatenate([np.asarray(c, float), np.asarray(h, float), np.asarray(rows, float).reshape(9)])


def many_as_few(rb, ev, Q):
    valid = P.prrtc_check_states(rb, ev, Q)
    few = np.concatenate([P.prrtc_check_states(rb, ev, Q[k:k + 1000]) for k in range(0, len(Q), 1000)])
    np.testing.assert_array_equal(valid, few)
    return valid


def test_short_rows_reach_past_the_box():
    """Rows of length 0.999: the test's face lies at half / 0.999, half a millimetre out."""
    robot = H.point_robot(lo=-2.0, hi=2.0)  # a sphere of 2 cm
    ev = P.make_env(H.scene(boxes=[box([0.1, 0.0, 0.5], [0.5, 0.5, 0.5], np.diag([0.999, 0.999, 1.0]))]))
    rng = np.random.default_rng(0)
    Q = np.stack([0.1 + rng.uniform(0.52015, 0.52045, N), rng.uniform(-0.4, 0.4, N)], 1).astype(np.float32)
    assert not many_as_few(P.make_robot(robot), ev, Q).any()


@pytest.mark.parametrize("decimals", [2, 3, 4])
def test_rotations_rounded_to_decimals(decimals):
    scene = turned_boxes(6, decimals)
    scene.boxes[:, 6:] = np.round(scene.boxes[:, 6:].astype(np.float64), decimals).astype(np.float32)
    scene.boxes[:, 3:6] *= 3.0
    robot = W.arm7()
    Q = np.random.default_rng(1).uniform(robot.lower, robot.upper, (N, robot.dof)).astype(np.float32)
    valid = many_as_few(P.make_robot(robot), P.make_env(scene), Q)
    assert 0 < valid.sum() < N


def test_moved_obstacles():
    robot = W.arm7()
    sc = W.scene_random_boxes(3, 4)
    obstacles = P.obstacles_from_scene(sc)
    rb, ev = P.make_robot(robot), P.make_env(sc)
    Q = np.random.default_rng(2).uniform(robot.lower, robot.upper, (N, robot.dof)).astype(np.float32)
    first = many_as_few(rb, ev, Q)
    far = W.scene_random_boxes(9, 4)
    far.boxes[:, :3] += [0.0, 0.0, 0.4]
    moved = P.obstacles_from_scene(far)
    with pytest.raises(P.PrrtcError):  # the second id does not exist: neither moves
        ev.update([0, 99], [moved[0], moved[1]])
    np.testing.assert_array_equal(many_as_few(rb, ev, Q), first)
    ev.update([1], [moved[1]])
    ev.update([0, 2, 3], [moved[0], moved[2], moved[3]])
    now = many_as_few(rb, ev, Q)
    np.testing.assert_array_equal(now, P.prrtc_check_states(rb, P.make_env(far), Q))
    assert (now != first).any()
