"""GPU parity of the list strategy where it can go wrong: tile edges, a threshold bin longer than its list, ties, a
sample that misleads in either direction, keys without low bits, lists longer than a block's shared memory."""
import numpy as np
import pytest
import torch

import oracle
import synth

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    import paper_2506_16235_b200 as nsml
    from gpu_util import (assert_payload_equal, check_compress, gpu_compress, mask_words, oracle_compress, sampled_elements,
                          took_the_fallback, to_device_grad)


def gauss(n, seed, spread=2.0):
    rng = np.random.default_rng(seed)
    return (rng.standard_normal(n) * 10.0 ** rng.uniform(-4.0, -4.0 + spread, n)).astype(np.float32)


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("n", [97 * 4096 - 1, 97 * 4096, 97 * 4096 + 1, 113 * 4096 + 513, 128 * 4096 + 1])
def test_tile_and_group_edges(n, dtype):
    g = gauss(n, n)
    g[-2:] = [3.0, -4.0]
    g[4095:4097] = [5.0, -6.0]
    if dtype == "bf16":
        g = synth.f32_to_bf16_bits(g)
    mask = np.random.default_rng(n).random(n) < 0.3
    for ratio, bits in ((0.002, 8), (0.03, 32), (0.2, 16)):
        check_compress(g, ratio, bits)
        check_compress(g, ratio, bits, mask_bool=mask)


@pytest.mark.parametrize("ties", [1, 1023, 1024, 1025, 40_000])
def test_threshold_bin_at_the_length_of_its_list(ties):
    # `ties` equal magnitudes around the threshold, spread over the bucket; half of them survive
    n, ratio = 1_000_003, 0.05
    rng = np.random.default_rng(ties)
    g = (rng.standard_normal(n) * 1e-3).astype(np.float32)
    k = nsml.nsml_k_of(n, ratio)
    order = rng.permutation(n)
    g[order[:k - (ties + 1) // 2]] = (2.0 + rng.random(k - (ties + 1) // 2)).astype(np.float32)
    g[order[k - (ties + 1) // 2:k - (ties + 1) // 2 + ties]] = np.float32(0.712345) * rng.choice(np.array([-1, 1], np.float32), ties)
    check_compress(g, ratio, 8)


def test_many_close_keys_in_the_threshold_bin():
    # 200k keys inside a few thousand float32 steps of one another: the bin is refined
    n = 2_000_000
    rng = np.random.default_rng(5)
    g = (rng.standard_normal(n) * 1e-4).astype(np.float32)
    where = rng.choice(n, 200_000, replace=False)
    g[where] = (np.float32(0.5).view(np.uint32) + rng.integers(0, 3000, 200_000).astype(np.uint32)).view(np.float32)
    for ratio in (0.05, 0.0995):
        check_compress(g, ratio, 16)


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_misleading_samples(dtype):
    n = 1 << 20
    rng = np.random.default_rng(3)
    keys = 4 if dtype == "f32" else 8
    conv = (lambda x: x) if dtype == "f32" else synth.f32_to_bf16_bits
    at = sampled_elements(n, keys)
    low = gauss(n, 1)
    low[at] = 0.0                     # the sample sees only zeros: everything non-zero is listed
    high = gauss(n, 2)
    high[at] *= np.float32(1e4)       # the sample sees only large values: too short a list
    hidden = gauss(n, 4)
    hidden[at] *= np.float32(1e-6)    # the sample sees only small values: the threshold lies above the window
    for g in (low, high, hidden):
        check_compress(conv(g), 0.01, 8)


def test_float32_bucket_widened_from_bfloat16():
    n = 3_000_001
    g = (synth.f32_to_bf16_bits(gauss(n, 8)).astype(np.uint32) << 16).view(np.float32)
    for ratio in (0.001, 0.02, 0.2):
        check_compress(g, ratio, 8)


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_list_longer_than_the_blocks_shared_memory(dtype):
    n = 20_000_003
    g = gauss(n, 9, spread=1.0)
    if dtype == "bf16":
        g = synth.f32_to_bf16_bits(g)
    for bits in (8, 16):
        check_compress(g, 0.24, bits)


def test_all_equal_large_bucket():
    g = np.full(2_000_001, 0.37, dtype=np.float32)
    check_compress(g, 0.05, 8)


@pytest.mark.parametrize("codes", [127, 3])
def test_quantised_gradient(codes):
    # few distinct magnitudes with full mantissas: the threshold's bin is one key with a great many ties
    n = 2_500_001
    rng = np.random.default_rng(codes)
    g = (np.rint(rng.standard_normal(n) * codes / 3).astype(np.float32) * np.float32(0.0123457))
    for ratio in (0.02, 0.2):
        check_compress(g, ratio, 8)


def test_equal_keys_beside_a_few_others_in_the_threshold_bin():
    # the bin overflows with one key, but holds others: found out while the list is read, and done over
    n, ratio = 1_000_003, 0.05
    rng = np.random.default_rng(11)
    g = (rng.standard_normal(n) * 1e-3).astype(np.float32)
    k = nsml.nsml_k_of(n, ratio)
    order = rng.permutation(n)
    g[order[:k - 2000]] = (2.0 + rng.random(k - 2000)).astype(np.float32)
    g[order[k - 2000:k + 3000]] = np.float32(0.712345)
    late = np.sort(order[k - 2000:k + 3000])[-3:]
    g[late] = np.nextafter(np.float32(0.712345), np.float32(1))
    check_compress(g, ratio, 8)


def test_feedback_when_ties_fill_the_threshold_bin():
    n, ratio = 600_011, 0.05
    rng = np.random.default_rng(12)
    g = (np.rint(rng.standard_normal(n) * 2).astype(np.float32) * np.float32(0.0123457))
    from oracle.adaptive import error_feedback_step
    residual = torch.zeros(n, device="cuda")
    want = np.zeros(n, dtype=np.float32)
    for bits in (8, 16, 32):
        payload = nsml.nsml_compress_feedback(torch.from_numpy(g).cuda(), residual, ratio, bits)
        ref, want = error_feedback_step(g, want, ratio, bits)
        assert_payload_equal(payload, ref)
        assert np.array_equal(residual.cpu().numpy().view(np.uint32), want.view(np.uint32))


# one block, one cluster, the list (its ties settled at once; a list shorter than k), the bucket itself
@pytest.mark.parametrize("n,ratio,hidden", [(5000, 0.4, False), (100_003, 0.1, False), (700_001, 0.1, False), (1 << 20, 0.1, True),
                                            (900_001, 0.5, False)])
@pytest.mark.parametrize("bits", [8, 16, 32])
def test_feedback_takes_selected_negative_zeros_out(n, ratio, hidden, bits):
    # fewer non-zero sums than survivors, all zero sums -0.0: a selected one leaves +0.0 where the payload carries its sign
    from oracle.adaptive import error_feedback_step
    rng = np.random.default_rng(n + bits)
    g = rng.standard_normal(n).astype(np.float32)
    zero = rng.random(n) >= 0.5 * ratio
    if hidden:  # (the sampler sees no zero, so the list holds the sampled elements only)
        zero[:] = True
        zero[sampled_elements(n, 4)] = False
    g[zero] = -0.0
    mask = rng.random(n) < 0.2
    start = np.where(zero, np.float32(-0.0), np.float32(0.5)).astype(np.float32)
    words = torch.from_numpy(mask_words(mask).view(np.int32)).cuda()
    for masked in (False, True):
        residual, want = torch.from_numpy(start.copy()).cuda(), start
        for _ in range(2):
            payload = nsml.nsml_compress_feedback(torch.from_numpy(g).cuda(), residual, ratio, bits, prune_mask=words if masked else None)
            ref, want = error_feedback_step(g, want, ratio, bits, prune_mask_=mask if masked else None)
            assert_payload_equal(payload, ref)
            assert np.array_equal(residual.cpu().numpy().view(np.uint32), want.view(np.uint32))


# more NaN (or infinities) than survivors: the sample's bounds are then themselves keys of NaN
@pytest.mark.parametrize("word", [0x7FC00000, 0x7F810000, 0x7FFF0000, 0xFFC00000, 0x7F800000])
@pytest.mark.parametrize("share", [0.03, 0.6, 1.0])
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_many_nonfinite_values_are_reported_and_nothing_else_is_touched(dtype, share, word):
    n, ratio = 700_001, 0.02
    rng = np.random.default_rng(int(share * 100))
    clean = gauss(n, 6)
    bad = clean.view(np.uint32).copy()
    bad[rng.random(n) < share] = word
    bad = bad.view(np.float32)
    if dtype == "bf16":
        clean, bad = synth.f32_to_bf16_bits(clean), (bad.view(np.uint32) >> 16).astype(np.uint16)
    need, room = nsml.nsml_payload_bytes(n, ratio, 8), nsml.nsml_workspace_bytes(n)
    payload = torch.full((need + 4096,), 0xA5, dtype=torch.uint8, device="cuda")
    ws = torch.full((room + (1 << 20),), 0xA5, dtype=torch.uint8, device="cuda")
    residual = torch.zeros(n, device="cuda")
    for call in ("plain", "residual"):
        if call == "plain":
            nsml.nsml_compress(to_device_grad(bad), ratio, 8, payload=payload, workspace=ws)
        else:
            nsml.nsml_compress_feedback(to_device_grad(bad), residual, ratio, 8, payload=payload, workspace=ws)
        assert nsml.nsml_last_status(ws) == nsml.NSML_ERR_NONFINITE
        assert bool((payload[need:] == 0xA5).all()) and bool((ws[room:] == 0xA5).all())
    # and the workspace serves an ordinary call
    out = nsml.nsml_compress(to_device_grad(clean), ratio, 8, payload=payload, workspace=ws)
    assert nsml.nsml_last_status(ws) == 0
    assert_payload_equal(out, oracle_compress(clean, ratio, 8))


# buckets of more than 8192 tiles (float32: 33,554,432 elements, bfloat16 twice as many): the list counts candidates per
# group of two or four tiles.  even: a run of 128 list entries spans more tiles than one round of 64 covers; crowded: all
# of them in a few tiles; close: the threshold's bin overflows and is refined over the list.
@pytest.mark.parametrize("n,dtype,kind", [(33_554_433, "f32", "even"), (33_554_433, "f32", "crowded"), (33_554_433, "f32", "close"),
                                          (67_108_865, "bf16", "even"), (67_112_961, "f32", "crowded")])
def test_buckets_of_more_tiles_than_groups(n, dtype, kind):
    rng = np.random.default_rng(n)
    g = rng.standard_normal(n, dtype=np.float32)
    ratios = (0.00005, 0.01, 0.2)
    if kind == "crowded":
        g[n // 3:n // 3 + n // 50] *= np.float32(1000.0)
        g[-4097:] *= np.float32(1000.0)
    if kind == "close":
        ratios = (0.01,)
        g *= np.float32(1e-4)
        where = rng.choice(n, 600_000, replace=False)
        g[where] = (np.float32(0.5).view(np.uint32) + rng.integers(0, 3000, where.size).astype(np.uint32)).view(np.float32)
    raw = synth.f32_to_bf16_bits(g) if dtype == "bf16" else g
    wants = oracle.compress_many(oracle.widen_bf16(raw) if dtype == "bf16" else g, ratios, 8)
    grad, ws = to_device_grad(raw), nsml.alloc_bytes(nsml.nsml_workspace_bytes(n), "cuda")
    for ratio, want in zip(ratios, wants):
        payload = nsml.nsml_compress(grad, ratio, 8, workspace=ws)
        assert nsml.nsml_last_status(ws) == 0
        assert took_the_fallback(ws) == (kind == "close")
        assert_payload_equal(payload, want)


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_feedback_on_more_tiles_than_groups(dtype):
    from oracle.adaptive import error_feedback_step
    n = 33_554_433 + 5000
    rng = np.random.default_rng(n)
    g = rng.standard_normal(n, dtype=np.float32)
    raw = g
    if dtype == "bf16":
        raw = synth.f32_to_bf16_bits(g)
        g = oracle.widen_bf16(raw)
    start = rng.standard_normal(n, dtype=np.float32)
    residual = torch.from_numpy(start.copy()).cuda()
    payload = nsml.nsml_compress_feedback(to_device_grad(raw), residual, 0.01, 16)
    want, left = error_feedback_step(g, start, 0.01, 16)
    assert_payload_equal(payload, want)
    assert np.array_equal(residual.cpu().numpy().view(np.uint32), left.view(np.uint32))
