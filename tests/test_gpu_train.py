"""The encoder's training kernels at the sizes where their work split changes:
sequences around the five groups of a CTA, batches around the part in which a
large batch is worked through (3420 triples on 152 SMs), one sequence per
weight-gradient CTA and dozens.

Tolerance: a sequence's forward and data gradients do not depend on which other
sequences are in the batch, so only the FP32 sums over the sequences differ in
order: at most 14,000 terms, 14,000 * 2^-24 relative to their absolute sum in the worst
case, sqrt of that in the expected one; 2e-5 of the gradient's norm."""
import numpy as np
import pytest

from paper_1812_10302_gb300 import dtws, synth, train

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def triples():
    m, n, B = 256, 400_000, 7001
    x = synth.walk_with_bursts(n, 31, 32, 33)
    rng = np.random.default_rng(3)
    q = rng.integers(0, n - m + 1, B)
    c = np.where(rng.random(B) < 0.5, np.clip(q + rng.integers(-20, 21, B), 0, n - m), rng.integers(0, n - m + 1, B))
    y = 10.0 ** rng.uniform(-3, 0, B)
    return train.load_weights(), dtws.enc_prep(x, q, m), dtws.enc_prep(x, c, m), y.astype(np.float32)


@pytest.mark.parametrize("rows", [1, 4, 5, 6, 759, 760, 761, 1523])
def test_forward_does_not_depend_on_the_batch(triples, rows):
    p, u = triples[0], triples[1]
    e = dtws.enc_forward(p, u[:rows])
    pick = sorted({0, rows // 2, rows - 1})
    for i in pick:
        np.testing.assert_array_equal(e[i], dtws.enc_forward(p, u[i:i + 1])[0])


@pytest.mark.parametrize("batch", [1, 2, 3, 76, 77, 3419, 3420, 3421, 7001])
def test_gradient_does_not_depend_on_the_order_of_the_batch(triples, batch):
    """(The pieces of a batch are no reference: the data gradients are scaled
    by one over the batch before they are rounded to BF16.)"""
    import torch
    p, uq, uc, y = triples[0], triples[1][:batch], triples[2][:batch], triples[3][:batch]
    loss, grad = dtws.enc_loss_grad(p, uq, uc, y)
    perm = np.random.default_rng(batch).permutation(batch)
    pl, pg = dtws.enc_loss_grad(p, uq[perm], uc[perm], y[perm])
    assert abs(loss - pl) <= 2e-5 * loss
    assert np.linalg.norm(grad - pg) <= 2e-5 * np.linalg.norm(grad)
    # the loss is the mean over the batch, whatever its parts
    cuts = list(range(0, batch, 1000)) + [batch]
    parts = [dtws.enc_loss_grad(p, uq[a:b], uc[a:b], y[a:b])[0] * (b - a) / batch for a, b in zip(cuts, cuts[1:])]
    assert abs(loss - sum(parts)) <= 2e-5 * loss
    # inputs on the device are read where they are
    dl, dg = dtws.enc_loss_grad(*(torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (p, uq, uc, y)))
    assert abs(dl - loss) <= 2e-5 * loss
    assert np.linalg.norm(dg - grad) <= 2e-5 * np.linalg.norm(grad)


@pytest.mark.parametrize("rows", [151, 152, 153, 303, 305, 1521])
def test_sequences_around_the_number_of_sms(triples, rows):
    """Sequences go to the SMs first, then to the groups of each: none is left
    out where their number passes the SMs' (152)."""
    p, u = triples[0], triples[1][:rows]
    e = dtws.enc_forward(p, u)
    some = np.unique(np.linspace(0, rows - 1, 40).astype(int))
    np.testing.assert_array_equal(e[some], np.concatenate([dtws.enc_forward(p, u[i:i + 1]) for i in some]))
