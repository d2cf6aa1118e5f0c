"""Edges of the mask build: tiles and units, the bracket's ends, the threshold's bin, misleading samples."""
import numpy as np
import pytest

from test_gpu_adaptive import check_mask
from gpu_util import sampled_elements

pytestmark = pytest.mark.gpu


def weights(n, seed):
    rng = np.random.default_rng(seed)
    return (rng.standard_normal(n) * 10.0 ** rng.uniform(-3, 0, n)).astype(np.float32)


# around a tile of the pass (4096), a unit of the select (8192), the first sampled size (16384)
@pytest.mark.parametrize("n", [1, 31, 33, 4095, 8191, 8193, 16383, 16384, 16385, 20_481, 3 * 4096 + 16384 - 1, 1_000_003])
def test_sizes(n):
    w = weights(n, n)
    for ratio in (0.001, 0.3, 0.97, 0.9995):  # (the last: nothing, or a handful, is pruned)
        check_mask(w, ratio)


@pytest.mark.parametrize("n", [70_001, 1 << 20])
@pytest.mark.parametrize("fill", [1e-9, 1e9])
def test_misleading_sample(n, fill):
    w = weights(n, 7)
    pos = sampled_elements(n, 4)
    w[pos] = fill * (1.0 + np.random.default_rng(8).random(pos.size))
    for ratio in (0.01, 0.5):
        check_mask(w, ratio)


@pytest.mark.parametrize("close", [900, 1024, 1025, 5000, 200_000])
def test_threshold_bin_around_the_keys_it_ranks(close):
    # `close` neighbouring keys, then the same number of equal ones, in the middle of the magnitudes
    n = 600_001
    w = weights(n, close)
    at = np.random.default_rng(close + 1).choice(n, close, replace=False)
    middle = np.sort(np.abs(w))[n // 2 - 50]
    for keys in (middle.view(np.uint32) + np.arange(close, dtype=np.uint32) % 700, np.full(close, middle.view(np.uint32), np.uint32)):
        w[at] = keys.view(np.float32) * np.where(at % 2, -1, 1).astype(np.float32)
        for ratio in (0.01, 0.0001):
            check_mask(w, ratio)


def test_bins_of_a_very_large_bucket_are_split_again():
    n = 200_000_000
    rng = np.random.default_rng(3)
    w = rng.standard_normal(n, dtype=np.float32)
    check_mask(w, 0.05)
