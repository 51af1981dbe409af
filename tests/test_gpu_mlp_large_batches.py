"""Gradients of batches of thousands of samples, whose products leave the clusters (more splits of K than a
cluster takes, more tiles than a wave).

A batch of 2^k copies of one sample has its gradients.  The head's are equal bit for bit: its operands are the
sample's over 2^k, and each range of K adds up a power of two of equal products of 16 significant bits.  The
layers before it see a row of dZ rounded to BF16 after FP32 sums in another order: each rounding moves a number
by at most 2^-9, two of them differ by 2^-8, over three layers 3 2^-8 < 2^-6 of a layer's norm."""
import numpy as np
import pytest

from paper_2503_06757_gb300 import prrtc as P
from paper_2503_06757_gb300 import workload as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2503_06757_gb300 import build
    build.build()


@pytest.mark.parametrize("name,batch", [("arm7", 4096), ("dual14", 4096), ("arm7", 8192), ("arm7", 16384)])
def test_copies_of_one_sample(name, batch):
    rb = W.ROBOTS[name]()
    init = W.proposal_init(rb.dof, 21)
    prop = P.Proposal(rb.dof, rb.lower, rb.upper,
                      np.concatenate([np.concatenate([w.ravel(), b]) for w, b in init]).astype(np.float32))
    rng = np.random.default_rng(4)
    occ = (rng.random((1, 4096)) < 0.1).astype(np.uint8)
    data = [rng.uniform(rb.lower, rb.upper, (1, rb.dof)).astype(np.float32) for _ in range(3)]
    rows = lambda a: np.repeat(a, batch, axis=0)
    loss1, one = prop.loss_and_grads(occ, *data)
    loss, g = prop.loss_and_grads(rows(occ), *[rows(a) for a in data])
    assert abs(loss - loss1) <= batch * 2.0 ** -24 * abs(loss1)
    at = 0
    for l, (w, b) in enumerate(init):
        a, r = g[at:at + w.size].astype(np.float64), one[at:at + w.size].astype(np.float64)
        if l == 3:
            np.testing.assert_array_equal(a, r)
        assert np.linalg.norm(a - r) <= 2.0 ** -6 * np.linalg.norm(r), l
        at += w.size + b.size
    losses = prop.train(occ, np.zeros(batch, np.int32), *[rows(a) for a in data], batch=batch, steps=2, lr=1e-3, seed=1)
    assert losses[1] < losses[0]
