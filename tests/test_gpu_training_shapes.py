"""The training kernels at the edges of their work split: one to 512 blocks of
128 samples (four, two and one CTA per block), and pair counts around the scaling kernel's 2048 pairs per block."""
import numpy as np
import pytest

from paper_1010_1486_gb300 import learn, su2

pytestmark = pytest.mark.gpu


def _pairs(n, seed):
    rng = np.random.default_rng(seed)
    bk = np.clip(rng.normal(12.0, 3.0, n), 3.0, 30.0)
    return np.stack([bk, np.clip(1.0 - rng.gamma(1.5, size=n) / bk, -1.0, 1.0)], axis=1).astype(np.float32)


def _trainer(seed):
    w = learn.initial_weights(seed)
    w[1120:1920] *= 10.0
    return su2.su2_trainer_create(w, 1)


@pytest.mark.parametrize("blocks", [1, 38, 39, 76, 77, 512])
def test_gradient_is_the_mean_of_its_blocks(blocks):
    """Rows of a block are summed in order and blocks in order, in binary32:
    the mean over n blocks differs from the binary64 mean of the blocks' own
    gradients by at most n roundings of the running sum."""
    torch = pytest.importorskip("torch")
    dev = torch.from_numpy(_pairs(128 * blocks, blocks)).cuda()
    tr = _trainer(blocks)
    try:
        su2.su2_trainer_set_input_scaling(tr, dev.data_ptr(), dev.shape[0])
        loss, grad = su2.su2_trainer_gradient(tr, dev.data_ptr(), dev.shape[0])
        parts = [su2.su2_trainer_gradient(tr, dev[128 * b:].data_ptr(), 128) for b in range(blocks)]
    finally:
        su2.su2_trainer_destroy(tr)
    each = np.stack([g.astype(np.float64) for _, g in parts])
    bound = (blocks + 2) * 2.0 ** -24 * np.abs(each).sum(axis=0) / blocks
    assert np.isfinite(grad).all() and np.abs(grad).max() > 0
    assert np.all(np.abs(grad - each.mean(axis=0)) <= bound + 1e-30)
    assert abs(loss - np.mean([l for l, _ in parts])) <= (blocks + 2) * 2.0 ** -24 * np.mean([abs(l) for l, _ in parts])


@pytest.mark.parametrize("n", [2, 255, 2048, 2049, 100_003, 400_000])
def test_input_scaling(n):
    torch = pytest.importorskip("torch")
    pairs = _pairs(n, n)
    dev = torch.from_numpy(pairs).cuda()
    tr = _trainer(3)
    try:
        for _ in range(2):  # the second call finds the ticket re-armed
            su2.su2_trainer_set_input_scaling(tr, dev.data_ptr(), n)
            w = su2.su2_trainer_get_weights(tr)
            x = pairs[:, 0].astype(np.float64)
            # one rounding to binary32 of each value, binary64 sums before it
            assert abs(w[1945] - x.mean()) <= 2.0 ** -23 * abs(x.mean())
            assert abs(w[1946] * x.std() - 1.0) <= 2.0 ** -22
    finally:
        su2.su2_trainer_destroy(tr)
