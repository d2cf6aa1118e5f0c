"""The select that works on the bucket itself where the sample gives no lower bound or one value fills the bucket: thresholds
that are zero, everything kept, ties by the million, magnitudes below the sample's bins.  Results against the oracle, and
the time of such calls beside that of an ordinary one."""
import numpy as np
import pytest
import torch

import oracle
import synth

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    import paper_2506_16235_b200 as nsml
    from gpu_util import assert_payload_equal, check_compress, mask_words, sampled_elements, to_device_grad

ROW = 148 * 4096  # elements of a row of segments on 148 SMs


def spread(n, seed):
    rng = np.random.default_rng(seed)
    return (rng.standard_normal(n) * 10.0 ** rng.uniform(-4, -1, n)).astype(np.float32)


def with_zeros(n, zeros, seed, rows=False):
    """`zeros` of the n elements are zero (of either sign): anywhere, or in runs of 768."""
    g, rng = spread(n, seed), np.random.default_rng(seed + 1)
    g[g == 0] = 1e-3
    at = rng.permutation(n)[:zeros]
    if rows:
        whole = n // 768
        picked = rng.permutation(whole)[:zeros // 768]
        at = (picked[:, None] * 768 + np.arange(768)).reshape(-1)
    g[at] = np.where(rng.random(at.size) < 0.5, np.float32(0.0), np.float32(-0.0))
    return g


def as_type(g, dtype):
    return synth.f32_to_bf16_bits(g) if dtype == "bf16" else g


@pytest.mark.parametrize("rows", [False, True])
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_more_kept_than_are_not_zero(dtype, rows):
    n = 2 * ROW + 4096 + 131
    g = as_type(with_zeros(n, int(0.7 * n), 20, rows), dtype)
    mask = np.random.default_rng(21).random(n) < 0.3
    for ratio in (0.35, 0.5, 0.9999):
        check_compress(g, ratio, 8)
        check_compress(g, ratio, 16, mask_bool=mask)


@pytest.mark.parametrize("off", [-700, -1, 0, 1, 700])
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_about_as_many_kept_as_are_not_zero(dtype, off):
    n = ROW + 999
    g = as_type(with_zeros(n, n // 2, 22), dtype)
    nonzero = n - n // 2
    check_compress(g, (nonzero + off - 0.5) / n, 32)


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("bits", [8, 16, 32])
def test_everything_kept(dtype, bits):
    for n, zeros in ((163_841, 0), (ROW, 1), (ROW + 130, ROW + 130), (2 * ROW + 5, ROW)):
        g = as_type(with_zeros(n, zeros, n), dtype)
        check_compress(g, 1.0, bits)
        check_compress(g, 1.0 - 1.0 / n, bits)  # all but one
        check_compress(g, 0.9999, bits, mask_bool=np.random.default_rng(3).random(n) < 0.1)


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_one_value_or_a_few(dtype):
    n = 2 * ROW + 1234
    rng = np.random.default_rng(24)
    signs = rng.choice(np.array([-1, 1], np.float32), n)
    quantised = (np.round(rng.standard_normal(n) * 4) / 64).astype(np.float32)
    for g in (np.zeros(n, np.float32), np.full(n, 0.0123, np.float32) * signs, quantised):
        for ratio in (0.13, 0.26, 0.5, 0.93):
            check_compress(as_type(g, dtype), ratio, 8)


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("ties", [3, 2000, 9000])
def test_one_bin_that_the_lists_hold(dtype, ties):
    # the window's keys fit the warps' lists, and a value repeated in it fills a bin beyond what is added key by key
    n = 2 * ROW + 321
    g = np.random.default_rng(33).standard_normal(n).astype(np.float32)
    order = np.argsort(-np.abs(g), kind="stable")
    at = n * 3 // 10
    g[order[at - ties // 2:at + ties - ties // 2]] = np.abs(g[order[at]])
    for k in (at - ties // 2, at - ties // 2 + 1, at, at + ties - ties // 2, at + ties):
        check_compress(as_type(g, dtype), (k - 0.5) / n, 8)


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_magnitudes_below_the_sample_bins(dtype):
    n = ROW + 77
    tiny = (np.random.default_rng(25).standard_normal(n) * 1e-20).astype(np.float32)
    check_compress(as_type(tiny, dtype), 0.5, 32)
    mixed = np.where(np.arange(n) % 3 == 0, spread(n, 26), tiny).astype(np.float32)
    mixed[::7] = 0.0
    for ratio in (0.2, 0.26, 0.3, 0.5, 0.8, 0.9):  # above, at and below the edge between the two, and among the zeros
        check_compress(as_type(mixed, dtype), ratio, 32)


@pytest.mark.parametrize("dtype,keys", [("f32", 4), ("bf16", 8)])
def test_samples_that_see_only_zeros_or_only_others(dtype, keys):
    n = 2 * ROW + 7
    at = sampled_elements(n, keys)
    for zeros_outside in (False, True):
        g = with_zeros(n, n // 4, 27)
        if zeros_outside:  # fewer than k keys that are not zero, which the sample does not see
            g[:] = 0.0
            g[at] = spread(at.size, 28)
        else:
            g[at] = 0.0
        for ratio in (0.3, 0.6):
            check_compress(as_type(g, dtype), ratio, 8)


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("ratio", [0.5, 1.0])
def test_residual_and_mask(dtype, ratio):
    from oracle.adaptive import error_feedback_step
    n = ROW + 4096 + 131
    raw = as_type(with_zeros(n, int(0.7 * n), 29, rows=True), dtype)
    g = oracle.widen_bf16(raw) if dtype == "bf16" else raw
    start = np.where(np.random.default_rng(30).random(n) < 0.1, spread(n, 31), 0.0).astype(np.float32)
    mask = np.random.default_rng(32).random(n) < 0.2
    residual = torch.from_numpy(start.copy()).cuda()
    mw = torch.from_numpy(mask_words(mask).view(np.int32)).cuda()
    payload = nsml.nsml_compress_feedback(to_device_grad(raw), residual, ratio, 8, prune_mask=mw)
    want, left = error_feedback_step(g, start, ratio, 8, prune_mask_=mask)
    assert_payload_equal(payload, want)
    assert np.array_equal(residual.cpu().numpy().view(np.uint32), left.view(np.uint32))


def test_time_beside_an_ordinary_call():
    # counted one by one at one address, 8M equal keys take 8 ms; an ordinary call of this size takes less than 0.1
    n = 8_000_000
    normal = torch.randn(n, device="cuda")
    rows = normal.clone()
    rows[: n // 768 * 768].view(-1, 768)[torch.rand(n // 768, device="cuda") < 0.54] = 0.0
    half = normal.clone()
    half[torch.rand(n, device="cuda") < 0.5] = 0.71875
    payload = nsml.alloc_bytes(nsml.nsml_payload_bytes(n, 1.0, 16), "cuda")
    ws = nsml.alloc_bytes(nsml.nsml_workspace_bytes(n), "cuda")

    def micros(g, ratio):
        times = []
        for _ in range(7):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            nsml.nsml_compress(g, ratio, 16, payload=payload, workspace=ws)
            b.record()
            torch.cuda.synchronize()
            times.append(a.elapsed_time(b) * 1e3)
        return sorted(times)[3]

    micros(normal, 0.5)
    ordinary = micros(normal, 0.5)
    for name, g, ratio in (("54 % zeros", rows, 0.5), ("all zero", torch.zeros_like(normal), 0.5), ("one value", torch.full_like(normal, 0.0123), 0.5),
                           ("half one value", half, 0.3), ("few values", torch.round(normal * 4) / 64, 0.5),
                           ("tiny", normal * 1e-20, 0.5), ("everything", normal, 1.0), ("nearly everything", normal, 0.99999)):
        took = micros(g, ratio)
        assert took <= 4 * ordinary, f"{name}: {took:.0f} us, an ordinary call {ordinary:.0f}"
