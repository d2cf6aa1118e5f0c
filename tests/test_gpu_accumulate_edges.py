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


# The partition reads payloads of few entries (16,384 per block) as a whole, four entries per thread: numbers of entries
# around a quad, a warp and a block; gaps of one, a few and all tiles; the first and the last tiles empty; long payloads of 64
# workers, which are searched, beside short ones; both sides of the line, workers on different sides of it in one call.
def _payload(n, idx, bits, seed):
    rng = np.random.default_rng(seed)
    k = idx.size
    vals = rng.standard_normal(k).astype(np.float32)
    if bits == 32:
        return nsml.pack_payload(n, 32, idx, f32=vals), vals.astype(np.float64)
    half = vals.astype(np.float16)
    return nsml.pack_payload(n, 16, idx, half=half.view(np.uint16)), half.astype(np.float64)


def _check_sum(n, index_sets, zero_first=True, sized=False):
    want = np.zeros(n) if zero_first else np.full(n, 0.5)
    payloads, most = [], 1.0
    for w, idx in enumerate(index_sets):
        raw, vals = _payload(n, np.asarray(idx, dtype=np.uint32), 16 if w % 2 else 32, w)
        want[np.asarray(idx, dtype=np.int64)] += vals
        most = max(most, float(np.abs(vals).max()))
        payloads.append(torch.from_numpy(raw).cuda())
    dense = torch.full((n,), 0.5, device="cuda")
    ws = torch.full((nsml.nsml_accumulate_workspace_bytes(n, len(payloads)),), 0xFF, dtype=torch.uint8, device="cuda")
    nsml.nsml_decompress_accumulate(payloads, dense, zero_first=zero_first, workspace=ws, sized=sized)
    assert nsml.nsml_last_status(ws) == 0
    # W float32 adds: at most W - 1 roundings of a running sum of at most W * most
    bound = len(payloads) ** 2 * most * 2.0 ** -24 + 1e-12
    assert float(np.abs(dense.cpu().numpy().astype(np.float64) - want).max()) <= bound


@pytest.mark.parametrize("n", [5000, 300_001, 3_000_001])
@pytest.mark.parametrize("sized", [False, True])
def test_partition_reads_whole_payloads(n, sized):
    rng = np.random.default_rng(n)
    sizes = [1, 2, 3, 4, 5, 127, 128, 129, 4095, 4096, 4097]
    sets = [np.sort(rng.choice(n, k, replace=False)) for k in sizes if k < n]
    _check_sum(n, sets, sized=sized)
    _check_sum(n, sets, zero_first=False, sized=sized)
    tail = min(n, 1000)
    gaps = [np.arange(tail), np.arange(n - tail, n), np.r_[0, n - 1], np.r_[0, 1, n // 2, n - 2, n - 1],
            np.arange(0, n, max(1, n // 37)), np.r_[np.arange(tail // 2), np.arange(n - tail // 2, n)]]
    _check_sum(n, gaps, sized=sized)


def test_partition_on_both_sides_of_its_line():
    n, W, line = 400_000, 64, (8 << 20) // 64
    rng = np.random.default_rng(4)
    for sizes in ([line] * W, [line + 1] * W, [line - 1 + w % 3 for w in range(W)], [line * 2 if w % 2 else 77 for w in range(W)]):
        _check_sum(n, [np.sort(rng.choice(n, k, replace=False)) for k in sizes])


def _line(n, W, many_calls=False):
    """Entries up to which a payload is read as a whole: 16,384 per block that the sum launches for a worker (sizes not
    told, or larger than an 8th of the bucket: as many blocks as there may be)."""
    blocks = max(1, min(64, 128 // W))
    return 16_384 * ((blocks + 3) // 4 if many_calls else blocks)


@pytest.mark.parametrize("sized", [False, True])
@pytest.mark.parametrize("many_calls", [False, True])
@pytest.mark.parametrize("W,n", [(1, 4_300_000), (2, 4_300_000), (8, 1_100_000), (64, 140_000)])
def test_payloads_around_the_line_between_reading_and_searching(W, n, many_calls, sized):
    line = _line(n, W, many_calls)
    rng = np.random.default_rng(W)

    def payloads(sizes):
        return [np.sort(rng.permutation(n)[:k]) for k in sizes]

    nsml.nsml_set_list_block_candidates(8192 if many_calls else 4096)
    try:
        for extra in (-1, 0, 1):
            _check_sum(n, payloads([line + extra] * W), sized=sized)
        _check_sum(n, payloads([line + w % 3 - 1 for w in range(W)]), sized=sized)
        _check_sum(n, payloads([line + 4097 if w % 2 else 77 for w in range(W)]), zero_first=False, sized=sized)
    finally:
        nsml.nsml_set_list_block_candidates(4096)
