"""Training repeats itself: the tiles of a minibatch are added in a fixed order, whatever order their
blocks run in."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def fsm():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2101_07690_gb300 import build, fsm as f
    build.build()
    f.load()
    return f


def _data(n, seed):
    rng = np.random.default_rng(seed)
    X = rng.normal(1.0, 2.0, (n, 32)).astype(np.float32)
    return X, (np.sin(X[:, 0]) + 0.5 * X[:, 1] + rng.normal(0, 0.2, n)).astype(np.float32)


# one row, a part of a tile, whole tiles, a ragged last minibatch, and 1250 tiles on at most 1024 blocks
@pytest.mark.parametrize("n,batch,epochs", [(1, 1, 3), (31, 31, 4), (4000, 128, 3), (9000, 256, 3), (5003, 300, 3),
                                            (40000, 40000, 3)])
def test_two_fits_are_equal_bit_for_bit(fsm, n, batch, epochs):
    X, y = _data(n, 7)
    runs = []
    for _ in range(3):
        m = fsm.fsm_mlp_create(1)
        try:
            fsm.fsm_mlp_fit_norm(m, X)
            loss = fsm.fsm_mlp_train(m, X, y, epochs, batch, 3e-3, seed=2)
            grads, mse = fsm.fsm_mlp_gradients(m, X, y)
            runs.append((fsm.fsm_mlp_get_params(m), grads, np.float32(loss), np.float32(mse)))
        finally:
            fsm.fsm_mlp_free(m)
    for other in runs[1:]:
        for a, b in zip(runs[0], other):
            assert np.array_equal(a, b)


def test_gradient_is_the_rounded_sum_of_its_tiles(fsm):
    """Of 8 tiles of 32 rows: each tile's own gradient is that of a call with its rows, 8 times as large
    (a power of two, so exactly); the sum of the eight is rounded once."""
    X, y = _data(256, 3)
    m = fsm.fsm_mlp_create(4)
    try:
        fsm.fsm_mlp_fit_norm(m, X)
        whole, _ = fsm.fsm_mlp_gradients(m, X, y)
        tiles = [fsm.fsm_mlp_gradients(m, X[r:r + 32], y[r:r + 32])[0].astype(np.float64) / 8.0 for r in range(0, 256, 32)]
    finally:
        fsm.fsm_mlp_free(m)
    total = np.zeros_like(tiles[0])
    for t in tiles:
        total = total + t
    assert np.array_equal(whole, total.astype(np.float32))
