"""A run of optimiser steps in one call equals the same steps one call each, bit for bit: within a call a step's
features are written while the update before it still runs, and its weight gradients run beside the bias
gradients; a call of one step has neither.  Gradients and updates are deterministic.

The library takes its batches from a seeded permutation (std::shuffle with std::mt19937_64).  A small program
prints it, so that each single step gets the same rows in the same order."""
import os
import subprocess

import numpy as np
import pytest

from paper_2503_06757_gb300 import prrtc as P
from paper_2503_06757_gb300 import workload as W

pytestmark = pytest.mark.gpu

ORDER = r'''
#include <algorithm>
#include <cstdio>
#include <cstdlib>
#include <random>
#include <vector>
int main(int, char** v) {
  std::vector<int> order(std::atoi(v[1]));
  std::mt19937_64 rng(std::strtoull(v[2], nullptr, 10));
  for (size_t i = 0; i < order.size(); ++i) order[i] = (int)i;
  std::shuffle(order.begin(), order.end(), rng);
  for (int i : order) printf("%d\n", i);
}
'''


@pytest.fixture(scope="module")
def order(tmp_path_factory):
    from paper_2503_06757_gb300 import build
    build.build()
    d = tmp_path_factory.mktemp("order")
    src, exe = os.path.join(d, "order.cpp"), os.path.join(d, "order")
    with open(src, "w") as f:
        f.write(ORDER)
    subprocess.run(["g++", "-O1", "-std=c++17", src, "-o", exe], check=True)
    return lambda n, seed: np.array(subprocess.run([exe, str(n), str(seed)], capture_output=True, text=True,
                                                   check=True).stdout.split(), int)


def proposal(robot):
    init = W.proposal_init(robot.dof, 21)
    return P.Proposal(robot.dof, robot.lower, robot.upper,
                      np.concatenate([np.concatenate([w.ravel(), b]) for w, b in init]).astype(np.float32))


@pytest.mark.parametrize("name,batch,steps", [("arm7", 1, 6), ("arm7", 8, 5), ("arm7", 37, 5), ("arm7", 512, 6),
                                              ("dual14", 512, 4), ("arm7", 1024, 4), ("dual14", 1300, 3),
                                              ("arm7", 4096, 3)])
def test_steps_of_one_call_equal_calls_of_one_step(order, name, batch, steps):
    robot = W.ROBOTS[name]()
    rng = np.random.default_rng(batch)
    n = batch * steps
    occ = (rng.random((5, 4096)) < 0.2).astype(np.uint8)
    scene = rng.integers(0, 5, n).astype(np.int32)
    data = [rng.uniform(robot.lower, robot.upper, (n, robot.dof)).astype(np.float32) for _ in range(3)]
    one = proposal(robot)
    losses = one.train(occ, scene, *data, batch=batch, steps=steps, lr=1e-3, seed=9)
    again = proposal(robot)
    rows = order(n, 9)
    back = np.argsort(order(batch, 4))  # undoes the shuffle of a call of one step
    for t in range(steps):
        pick = rows[t * batch:(t + 1) * batch][back]
        loss = again.train(occ, scene[pick], *[d[pick] for d in data], batch=batch, steps=1, lr=1e-3, seed=4)
        assert abs(loss[0] - losses[t]) <= batch * 2.0 ** -22 * abs(losses[t])  # summed in any order
    np.testing.assert_array_equal(one.params(), again.params())
    np.testing.assert_array_equal(one.grads(), again.grads())
