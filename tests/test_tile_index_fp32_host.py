"""The tile-pair enumeration of auto counts below 32768 tiles (`item_to_tiles`), by
host emulation: there the row comes from an FP32 square root, with and without a
fused multiply-add, and is settled by comparisons of 32-bit products.  Every item
maps to its tile pair, no product leaves 32 bits, and the settling takes few steps."""
import numpy as np
import pytest

F = np.float32


def item_to_tiles(k, T, fused):
    """The kernel's steps for items k (int64 holding 32-bit values) of T tiles."""
    b = F(F(2) * F(T) + F(1))
    kf = (F(8) * k.astype(F)).astype(F)
    if fused:
        x = (np.float64(b) * np.float64(b) - kf.astype(np.float64)).astype(F)
    else:
        x = (F(b * b) - kf).astype(F)
    i = ((b - np.sqrt(np.maximum(x, F(0)))).astype(F) * F(0.5)).astype(F).astype(np.int64)
    i = np.clip(i, 0, T - 1)
    steps = np.zeros_like(i)
    top = 0
    while True:
        a, c = i * T, i * (i - 1)
        top = max(top, int(a.max()), int(c.max()))
        down = (i > 0) & (a - c // 2 > k)
        if not down.any():
            break
        i, steps = i - down, steps + down
    while True:
        a, c = (i + 1) * T, (i + 1) * i
        top = max(top, int(a.max()), int(c.max()))
        up = (i + 1 < T) & (a - c // 2 <= k)
        if not up.any():
            break
        i, steps = i + up, steps + up
    assert top < 2 ** 31, "a product leaves 32 bits"
    return i, i + (k - (i * T - i * (i - 1) // 2)), steps


@pytest.mark.parametrize("fused", [False, True])
@pytest.mark.parametrize("T", [1, 2, 3, 31, 32, 33, 100, 977, 1954, 5000, 9766, 16383, 23170,
                               32766, 32767])
def test_items_map_to_their_tile_pairs(T, fused):
    n = T * (T + 1) // 2
    assert 8 * n < 2 ** 32 + 2 ** 21 and n < 2 ** 29 + 2 ** 15
    I = np.arange(T, dtype=np.int64)
    start = I * T - I * (I - 1) // 2
    rng = np.random.default_rng(T)
    last = np.arange(max(0, n - 200000), n)
    for k in (start, start + (T - 1 - I), start[1:] - 1, rng.integers(0, n, 300000), last,
              np.arange(min(n, 200000))):
        if len(k) == 0:
            continue
        i, j, steps = item_to_tiles(k, T, fused)
        row = np.searchsorted(start, k, side="right") - 1
        assert np.array_equal(i, row) and np.array_equal(j, row + (k - start[row]))
        assert np.all((j >= i) & (j < T))
        assert int(steps.max()) <= 16, "an FP32 estimate far off its row"


def test_every_item_of_small_counts_once():
    for T in range(1, 70):
        n = T * (T + 1) // 2
        i, j, _ = item_to_tiles(np.arange(n), T, False)
        assert len(set(zip(i.tolist(), j.tolist()))) == n


def test_the_estimate_alone_would_not_do():
    T = 32767
    k = np.arange(T * (T + 1) // 2 - 4000, T * (T + 1) // 2)
    _, _, steps = item_to_tiles(k, T, False)
    assert steps.max() >= 1
