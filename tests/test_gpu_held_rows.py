"""Lockstep batches whose held rows come close to their limit: fewer workers run side by side, the plans stay
those of one round at a time, and the buffer stays within the limit."""
import numpy as np
import pytest

from paper_2503_06757_gb300 import prrtc as P
from paper_2503_06757_gb300 import workload as W
from tests.test_gpu_rounds import problems, same, shelf

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

LIMIT = 1 << 28  # floats


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2503_06757_gb300 import build
    build.build()


@pytest.mark.parametrize("workers", [1, 3])
def test_lockstep_below_the_limit(workers):
    robot = W.dual14()
    items = problems(robot, shelf(robot, 2), 70)
    kw = dict(mode=P.MODE_LOCKSTEP, workers=workers, max_iters=7, range=0.001, tree_capacity=4096, path_capacity=4096)
    span = np.linalg.norm(np.asarray(robot.upper) - np.asarray(robot.lower))
    rows = 70 * 16 * span / 0.001  # a worker's, at most three rows a problem fewer than the library's
    assert workers * rows < 0.9 * LIMIT < 1.1 * LIMIT < (16 // workers) * workers * rows
    want = P.prrtc_plan_batch(items, P.params(warps_per_block=workers, **kw))  # one round at a time
    before = torch.cuda.mem_get_info()[0]
    got = P.prrtc_plan_batch(items, P.params(**kw))
    assert before - torch.cuda.mem_get_info()[0] <= 4 * LIMIT + (1 << 26)
    for k in range(len(items)):
        same(got[k], want[k], (workers, k))


def test_serial_gives_large_scratch_back():
    """70 problems of steps of 0.01: 150 MB of held rows, of which at most 64 MiB stay."""
    robot = W.dual14()
    items = problems(robot, shelf(robot, 2), 70)
    kw = dict(mode=P.MODE_SERIAL, max_iters=3, tree_capacity=4096, path_capacity=4096)
    span = np.linalg.norm(np.asarray(robot.upper) - np.asarray(robot.lower))
    assert 1 << 27 < 4 * 16 * 70 * 16 * span / 0.01 < 1 << 28
    P.prrtc_plan_batch(items, P.params(**kw))  # arenas and the usual scratch
    before = torch.cuda.mem_get_info()[0]
    for _ in range(2):
        P.prrtc_plan_batch(items, P.params(range=0.01, **kw))
        assert before - torch.cuda.mem_get_info()[0] <= 1 << 26
