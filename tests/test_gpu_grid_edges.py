"""GPU parity of the select that works on the bucket itself (kept fractions from an eighth on) where it can go wrong:
edges of its segments and rows, buckets that its shared memory does not hold, a list of window keys that overflows, samples
that mislead, ties across slices, replay from a graph."""
import numpy as np
import pytest
import torch

import oracle
import synth

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    import paper_2506_16235_b200 as nsml
    from gpu_util import assert_payload_equal, check_compress, mask_words, oracle_compress, sampled_elements, to_device_grad


def spread(n, seed, lo=-4, hi=-1):
    rng = np.random.default_rng(seed)
    return (rng.standard_normal(n) * 10.0 ** rng.uniform(lo, hi, n)).astype(np.float32)


# A slice is 128 float32 (256 bfloat16) elements, a segment 32 of them, a row 148 segments: the ragged end in the first and
# in a later slice, a lone element, one and several rows.
SEG, ROW = 4096, 148 * 4096
SIZES = [163_841, 41 * SEG, 41 * SEG + 1, 41 * SEG + 127, 42 * SEG - 1, ROW - 1, ROW, ROW + 1, ROW + SEG + 129, 2 * ROW + 5 * SEG + 130,
         7 * ROW + 3]


@pytest.mark.parametrize("n", SIZES)
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_segment_and_row_edges(n, dtype):
    g = spread(n, n)
    g[-3:] = [3.0, -4.0, 5.0]
    mask = np.random.default_rng(n + 1).random(n) < 0.3
    if dtype == "bf16":
        g = synth.f32_to_bf16_bits(g)
    check_compress(g, 0.3, 8)
    check_compress(g, 0.7, 16, mask_bool=mask)
    check_compress(g, 0.13, 32)


@pytest.mark.parametrize("n", [163_841, ROW + SEG + 129, 5 * ROW + 77])
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("bits", [8, 16, 32])
def test_feedback_with_a_mask(n, dtype, bits):
    from oracle.adaptive import error_feedback_step
    g = spread(n, n + 2)
    raw = g
    if dtype == "bf16":
        raw = synth.f32_to_bf16_bits(g)
        g = oracle.widen_bf16(raw)
    mask = np.random.default_rng(3).random(n) < 0.25
    start = spread(n, 5)
    residual = torch.from_numpy(start.copy()).cuda()
    mw = torch.from_numpy(mask_words(mask).view(np.int32)).cuda()
    payload = nsml.nsml_compress_feedback(to_device_grad(raw), residual, 0.4, bits, prune_mask=mw)
    want, left = error_feedback_step(g, start, 0.4, bits, prune_mask_=mask)
    assert_payload_equal(payload, want)
    assert np.array_equal(residual.cpu().numpy().view(np.uint32), left.view(np.uint32))


# 20M float32 (30M bfloat16) elements are more than the blocks hold: slices are read again, with masks and residuals too
@pytest.mark.parametrize("kind", ["f32", "bf16", "masked", "feedback"])
def test_buckets_larger_than_the_shared_memory(kind):
    from oracle.adaptive import error_feedback_step
    n = 20_000_003 if kind != "bf16" else 30_000_003
    g = np.random.default_rng(6).standard_normal(n, dtype=np.float32)
    if kind == "feedback":
        start = np.random.default_rng(7).standard_normal(n, dtype=np.float32)
        residual = torch.from_numpy(start.copy()).cuda()
        payload = nsml.nsml_compress_feedback(torch.from_numpy(g).cuda(), residual, 0.5, 8)
        want, left = error_feedback_step(g, start, 0.5, 8)
        assert_payload_equal(payload, want)
        assert np.array_equal(residual.cpu().numpy().view(np.uint32), left.view(np.uint32))
    elif kind == "masked":
        check_compress(g, 0.5, 16, mask_bool=np.random.default_rng(8).random(n) < 0.25)
    else:
        check_compress(synth.f32_to_bf16_bits(g) if kind == "bf16" else g, 0.5, 8)


# One key on half of the elements, the threshold among them or beside them: the warps' lists of window keys overflow, the
# ties' last index lies in the first, a middle or the last slice.
@pytest.mark.parametrize("ratio", [0.1300001, 0.3, 0.6, 0.62999])
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_ties_that_overflow_the_lists(ratio, dtype):
    n = 3 * ROW + 1001
    rng = np.random.default_rng(9)
    g = spread(n, 10, -6, -3)
    order = rng.permutation(n)
    g[order[:n // 2]] = np.float32(0.71875) * rng.choice(np.array([-1, 1], np.float32), n // 2)
    g[order[n // 2:n // 2 + n // 8]] = 2.0 + rng.random(n // 8, dtype=np.float32)
    check_compress(synth.f32_to_bf16_bits(g) if dtype == "bf16" else g, ratio, 8)


def test_close_keys_need_another_histogram():
    n = 2 * ROW + 999  # 300,000 keys within 3000 units in the last place of each other around the threshold
    rng = np.random.default_rng(12)
    g = spread(n, 13, -6, -4)
    where = rng.choice(n, 300_000, replace=False)
    g[where] = (np.float32(0.5).view(np.uint32) + rng.integers(0, 3000, where.size).astype(np.uint32)).view(np.float32)
    for ratio in (0.15, 0.24):
        check_compress(g, ratio, 16)


@pytest.mark.parametrize("dtype,keys", [("f32", 4), ("bf16", 8)])
def test_misleading_samples(dtype, keys):
    n = 2 * ROW + 7
    at = sampled_elements(n, keys)
    conv = synth.f32_to_bf16_bits if dtype == "bf16" else (lambda x: x)
    for scale in (0.0, 1e4, 1e-6):  # the sample sees zeros; a bound too high (a second stream); the threshold above the window
        g = spread(n, 14)
        g[at] *= np.float32(scale)
        for bits in (8, 32):
            check_compress(conv(g), 0.3, bits)
    from oracle.adaptive import error_feedback_step
    g = spread(n, 15)
    g[at] *= np.float32(1e4)
    raw = conv(g)
    g = oracle.widen_bf16(raw) if dtype == "bf16" else g
    start = np.zeros(n, np.float32)
    residual = torch.zeros(n, device="cuda")
    payload = nsml.nsml_compress_feedback(to_device_grad(raw), residual, 0.3, 8)
    want, left = error_feedback_step(g, start, 0.3, 8)
    assert_payload_equal(payload, want)
    assert np.array_equal(residual.cpu().numpy().view(np.uint32), left.view(np.uint32))


def test_magnitudes_outside_the_sample_bins():
    n = 400_003  # far below and above the octaves that the sample tells apart
    for scale in (1e-30, 1e-38, 1e30):
        check_compress((spread(n, 16, -1, 0) * np.float32(scale)).astype(np.float32), 0.3, 32)


def test_replayed_from_a_graph_beside_another_stream():
    n = 3 * ROW + 11
    g = spread(n, 17)
    buf, side, other = to_device_grad(g), torch.cuda.Stream(), torch.cuda.Stream()
    buf2 = buf.clone()
    ws, ws2 = (nsml.alloc_bytes(nsml.nsml_workspace_bytes(n), "cuda") for _ in range(2))
    payload = nsml.alloc_bytes(nsml.nsml_payload_bytes(n, 0.5, 8), "cuda")
    nsml.nsml_compress(buf, 0.5, 8, payload=payload, workspace=ws)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=side):
        nsml.nsml_compress(buf, 0.5, 8, payload=payload, workspace=ws, stream=side)
    for rep in range(3):
        fresh = np.roll(g, 1234 * (rep + 1))
        buf.copy_(torch.from_numpy(fresh))
        torch.cuda.synchronize()
        graph.replay()
        eager = nsml.nsml_compress(buf2, 0.3, 16, workspace=ws2, stream=other)  # on another stream at the same time
        torch.cuda.synchronize()
        assert_payload_equal(payload, oracle_compress(fresh, 0.5, 8))
        assert_payload_equal(eager, oracle_compress(g, 0.3, 16))
        assert nsml.nsml_last_status(ws) == 0 and nsml.nsml_last_status(ws2) == 0
