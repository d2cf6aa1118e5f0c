"""GPU parity of the buckets that one block or one cluster holds in shared memory: at and around the switches between
one block, the cluster and the other strategies, with values that tie, and with a residual."""
import numpy as np
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    import paper_2506_16235_b200 as nsml
    from gpu_util import assert_payload_equal, check_compress, mask_words
    from oracle.adaptive import error_feedback_step

SIZES = [1, 127, 128, 129, 8191, 8192, 8193, 8 * 2176 + 1, 49_151, 8 * 20_480 - 1, 8 * 20_480, 8 * 20_480 + 1]


def values(kind, n):
    rng = np.random.default_rng(n)
    g = (rng.standard_normal(n) * 10.0 ** rng.uniform(-4, -2, n)).astype(np.float32)
    if kind == "ties":
        g = np.rint(g * 2000).astype(np.float32)
    if kind == "sparse":
        g[rng.random(n) < 0.95] = 0.0
    return g


@pytest.mark.parametrize("kind", ["normal", "ties", "sparse"])
@pytest.mark.parametrize("n", SIZES)
def test_sizes(n, kind):
    g = values(kind, n)
    mask = np.random.default_rng(n + 1).random(n) < 0.3
    for ratio, bits in ((0.003, 16), (0.1, 8), (0.6, 32), (1.0, 8)):
        check_compress(g, ratio, bits)
    check_compress(g, 0.2, 8, mask_bool=mask)
    check_compress(synth.f32_to_bf16_bits(g), 0.3, 8, mask_bool=mask)


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("n", [5, 8192, 30_001])
def test_feedback(n, dtype):
    rng = np.random.default_rng(n)
    mask = rng.random(n) < 0.5
    residual = torch.zeros(n, device="cuda")
    want = np.zeros(n, dtype=np.float32)
    words = torch.from_numpy(mask_words(mask).view(np.int32)).cuda()
    for ratio, bits in ((0.05, 8), (0.7, 16), (0.1, 32), (0.9, 8)):  # (more than half: pruned parameters are selected)
        g = (rng.standard_normal(n) * 1e-2).astype(np.float32)
        if dtype == "bf16":
            raw = synth.f32_to_bf16_bits(g)
            g = (raw.astype(np.uint32) << 16).view(np.float32)
            dev = torch.from_numpy(raw.view(np.int16)).cuda().view(torch.bfloat16)
        else:
            dev = torch.from_numpy(g).cuda()
        payload = nsml.nsml_compress_feedback(dev, residual, ratio, bits, prune_mask=words)
        ref, want = error_feedback_step(g, want, ratio, bits, prune_mask_=mask)
        assert_payload_equal(payload, ref)
        assert np.array_equal(residual.cpu().numpy().view(np.uint32), want.view(np.uint32))


# the threshold's bin (a sixteenth of an octave) with as many keys as are looked at one per thread, one fewer and one more;
# all in one block's part or spread over the cluster's, distinct or equal
@pytest.mark.parametrize("n", [6000, 8192, 8193, 60_000])
@pytest.mark.parametrize("count", [1, 2, 1023, 1024, 1025])
@pytest.mark.parametrize("kind", ["spread", "together", "equal", "zeros"])
def test_keys_of_the_first_digits_bin(n, count, kind):
    rng = np.random.default_rng(n + count)
    g = (rng.random(n) * 1e-3 + 1e-6).astype(np.float32)
    order = np.arange(n) if kind == "together" else rng.permutation(n)
    if kind == "zeros":
        g[order[:count]] = 0.0  # (pruned parameters and empty rows share the lowest bin)
        ratios = [(n - count + take) / n for take in {1, (count + 1) // 2, count}]
    else:
        g[order[:count]] = 1.01 if kind == "equal" else 1.0 + rng.random(count) * 0.06
        g[order[count:count + 100]] = 8.0 + rng.random(100).astype(np.float32)
        ratios = [(100 + take) / n for take in {1, (count + 1) // 2, count}]
    g *= rng.choice(np.array([-1.0, 1.0], np.float32), n)
    for ratio in ratios:
        check_compress(g, ratio * (1 - 1e-9), 8)
