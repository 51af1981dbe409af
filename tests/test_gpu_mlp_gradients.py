"""Gradients of the learned proposal at the edges of the batch sizes.

A batch of 2^k copies of one sample has that sample's gradients exactly: every row's share is the sample's
over 2^k, a product of two BF16 numbers has 16 significant bits, and up to 128 equal ones (a power of two of
them beyond) add up exactly in FP32.  So every layer's weight gradients are equal bit for bit over the
numbers of K tiles and splits that the batch sizes bring.  A bias gradient adds up n FP32 numbers of 24 bits
one after the other, each sum rounded once: n 2^-24 of its size."""
import numpy as np
import pytest

from paper_2503_06757_gb300 import prrtc as P
from paper_2503_06757_gb300 import workload as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2503_06757_gb300 import build
    build.build()


@pytest.mark.parametrize("name", ["arm7", "dual14"])
def test_copies_of_one_sample_have_its_gradients(name):
    rb = W.ROBOTS[name]()
    init = W.proposal_init(rb.dof, 21)
    prop = P.Proposal(rb.dof, rb.lower, rb.upper,
                      np.concatenate([np.concatenate([w.ravel(), b]) for w, b in init]).astype(np.float32))
    rng = np.random.default_rng(4)
    occ = (rng.random((1, 4096)) < 0.1).astype(np.uint8)
    qs, qg, tg = (rng.uniform(rb.lower, rb.upper, (1, rb.dof)).astype(np.float32) for _ in range(3))
    rows = lambda a, n: np.repeat(a, n, axis=0)
    _, one = prop.loss_and_grads(occ, qs, qg, tg)
    assert np.count_nonzero(one) > one.size // 20
    for n in (2, 8, 32, 64, 128, 256, 512, 1024):
        _, g = prop.loss_and_grads(rows(occ, n), rows(qs, n), rows(qg, n), rows(tg, n))
        at = 0
        for w, b in init:
            np.testing.assert_array_equal(g[at:at + w.size], one[at:at + w.size], err_msg=str(n))
            at += w.size
            gb, ob = g[at:at + b.size].astype(np.float64), one[at:at + b.size].astype(np.float64)
            assert np.all(np.abs(gb - ob) <= n * 2.0 ** -24 * np.abs(ob)), n
            at += b.size
