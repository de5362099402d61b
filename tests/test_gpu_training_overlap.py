"""A fit queues its steps with overlapping launches: a step and its Adam update
are on the GPU while the ones before still write the weights and partial sums
that they read.  The same steps, one call each (and so each waited for), must
give the same losses and weights bit for bit, at one, two and four CTAs per 128
samples."""
import numpy as np
import pytest

from paper_1010_1486_gb300 import learn, su2

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("batch,steps", [(128, 400), (4096, 400), (76 * 128, 200), (16384, 100), (65536, 40)])
def test_overlapped_steps_equal_separate_ones(batch, steps):
    torch = pytest.importorskip("torch")
    rng = np.random.default_rng(batch)
    n = 50_000
    bk = np.clip(rng.normal(12.0, 3.0, n), 3.0, 30.0)
    pairs = np.stack([bk, np.clip(1.0 - rng.gamma(1.5, size=n) / bk, -1.0, 1.0)], axis=1).astype(np.float32)
    dev = torch.from_numpy(pairs).cuda()
    out = []
    for calls in ([steps], [1] * steps):
        tr = su2.su2_trainer_create(learn.initial_weights(5), 9)
        try:
            su2.su2_trainer_set_input_scaling(tr, dev.data_ptr(), n)
            losses = [su2.su2_trainer_fit(tr, dev.data_ptr(), n, k, batch) for k in calls]
            out.append((np.concatenate(losses), su2.su2_trainer_get_weights(tr)))
        finally:
            su2.su2_trainer_destroy(tr)
    (la, wa), (lb, wb) = out
    assert np.array_equal(la.view(np.uint32), lb.view(np.uint32))
    assert np.array_equal(wa.view(np.uint32), wb.view(np.uint32))
    assert np.isfinite(la).all() and la[-5:].mean() < la[:5].mean()


@pytest.mark.parametrize("n", [4095, 4096, 4097, 6145])
def test_input_scaling_either_side_of_one_block(n):
    torch = pytest.importorskip("torch")
    x = np.random.default_rng(n).normal(12.0, 3.0, n).astype(np.float32)
    dev = torch.from_numpy(np.stack([x, np.zeros_like(x)], axis=1)).cuda()
    tr = su2.su2_trainer_create(learn.initial_weights(5), 9)
    try:
        for _ in range(2):  # the second call finds the ticket re-armed
            su2.su2_trainer_set_input_scaling(tr, dev.data_ptr(), n)
            w = su2.su2_trainer_get_weights(tr)
            # one rounding to binary32 of each value, binary64 sums before it
            x64 = x.astype(np.float64)
            assert abs(w[1945] - x64.mean()) <= 2.0 ** -23 * abs(x64.mean())
            assert abs(w[1946] * x64.std() - 1.0) <= 2.0 ** -22
    finally:
        su2.su2_trainer_destroy(tr)
