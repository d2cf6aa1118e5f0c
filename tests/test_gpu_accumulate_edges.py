"""GPU parity of the sum at the edges of its tiles: the switch between the two tile sizes, the last (partial) tile,
quads that straddle a worker's range, ranges of more than one unit of 128 quads, many workers and empty ones."""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    import paper_2506_16235_b200 as nsml
    from gpu_util import check_accumulate, payload_to_device

SWITCH = 1024 * 2048  # largest bucket that takes the small tile


def crowded_payload(n, k, bits, seed):
    """k survivors, half of them in one short run of the bucket (several units of one tile), the rest anywhere."""
    rng = np.random.default_rng(seed)
    g = np.zeros(n, dtype=np.float32)
    run = min(n, max(1, k // 2))
    start = int(rng.integers(0, n - run + 1))
    g[start:start + run] = rng.standard_normal(run)
    g[rng.choice(n, size=min(n, k), replace=False)] += np.float32(3.0) + rng.random(min(n, k), dtype=np.float32)
    return oracle.compress(g, k / n, bits)


@pytest.mark.parametrize("zero_first", [True, False])
@pytest.mark.parametrize("n", [2047, 2048, 2049, SWITCH - 1, SWITCH, SWITCH + 1, SWITCH + 8191, 296 * 8192, 296 * 8192 + 1])
def test_tile_edges(n, zero_first):
    want = [crowded_payload(n, min(n, 20_011), bits, n + bits) for bits in (8, 16, 32)]
    init = None if zero_first else np.random.default_rng(1).standard_normal(n).astype(np.float32)
    check_accumulate([payload_to_device(p) for p in want], want, n, zero_first, dense_init=init)


@pytest.mark.parametrize("W", [33, 64])
def test_many_workers_most_of_them_sparse(W):
    n = 100_003
    want = [crowded_payload(n, 1 if w % 3 else 5000, 8, w) for w in range(W)]
    check_accumulate([payload_to_device(p) for p in want], want, n, zero_first=True)


def test_one_workspace_sized_for_the_largest_bucket_serves_them_all():
    # a gradient set in 25 MB buckets: the shorter ones need more room for their (smaller) tiles than the longest one
    W, sizes = 8, (6_553_600, 2_424_832, SWITCH, 2_000_000, 12_289)
    ws = nsml.alloc_bytes(nsml.nsml_accumulate_workspace_bytes(max(sizes), W), "cuda")
    for n in sizes:
        want = [crowded_payload(n, 1500, 8, n + w) for w in range(W)]
        dense = torch.full((n,), 7.0, device="cuda")
        nsml.nsml_decompress_accumulate([payload_to_device(p) for p in want], dense, workspace=ws)
        assert nsml.nsml_last_status(ws) == 0
        ref = oracle.decompress_sum(want, n)
        largest = max(float(np.abs(p.raw).max()) for p in want)
        assert float(np.abs(dense.cpu().numpy().astype(np.float64) - ref).max()) <= 1e-6 * largest
