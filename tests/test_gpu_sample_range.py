"""The sample's bounds at every magnitude a float can have: results of the list strategy and of the mask build, and that no
magnitude leaves a call without bounds."""
import numpy as np
import pytest
import torch

import oracle
import synth

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    import paper_2506_16235_b200 as nsml
    from gpu_util import assert_payload_equal, took_the_fallback, to_device_grad
    from test_gpu_adaptive import check_mask

# inside and at both edges of the octaves that are counted finely (2^-76 to 2^32), below, above, next to infinity and
# among the subnormal numbers
SCALES = [1.0, 2.0 ** -76, 2.0 ** 32, 2.0 ** -96, 1e-30, 1e-36, 1e-38, 1e-41, 1e12, 1e30, 2e37]


def values(n, seed, scale):
    rng = np.random.default_rng(seed)
    return (rng.standard_normal(n) * scale).astype(np.float32)


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("scale", SCALES)
def test_list_strategy(scale, dtype):
    n = 400_003
    g = values(n, 1, scale)
    raw = synth.f32_to_bf16_bits(g) if dtype == "bf16" else g
    wide = oracle.widen_bf16(raw) if dtype == "bf16" else g
    ws = nsml.alloc_bytes(nsml.nsml_workspace_bytes(n, nsml.NSML_BF16 if dtype == "bf16" else nsml.NSML_F32), "cuda")
    for ratio in (0.001, 0.05):
        payload = nsml.nsml_compress(to_device_grad(raw), ratio, 32, workspace=ws)
        assert nsml.nsml_last_status(ws) == 0
        assert_payload_equal(payload, oracle.compress(wide, ratio, 32))
        if scale in (1.0, 2.0 ** -76):  # (where bins are coarse, a short bucket's threshold bin may be too full)
            assert not took_the_fallback(ws)


@pytest.mark.parametrize("scale", SCALES)
def test_mask_build(scale):
    for ratio in (0.01, 0.6):
        check_mask(values(300_001, 2, scale), ratio)


def test_no_magnitude_costs_a_list_of_the_whole_bucket():
    n = 16_000_000
    normal = torch.randn(n, device="cuda")
    payload = nsml.alloc_bytes(nsml.nsml_payload_bytes(n, 0.01, 32), "cuda")
    ws = nsml.alloc_bytes(nsml.nsml_workspace_bytes(n), "cuda")

    def micros(g):
        times = []
        for _ in range(7):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            nsml.nsml_compress(g, 0.01, 32, payload=payload, workspace=ws)
            b.record()
            torch.cuda.synchronize()
            times.append(a.elapsed_time(b) * 1e3)
        return sorted(times)[3]

    micros(normal)
    ordinary = micros(normal)
    for scale in (1e-30, 1e-36, 1e12, 1e30):
        took = micros(normal * scale)
        assert took <= 2 * ordinary, f"{scale}: {took:.0f} us, an ordinary call {ordinary:.0f}"
