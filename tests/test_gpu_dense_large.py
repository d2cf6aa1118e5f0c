"""Compress of buckets of hundreds of millions of elements at high kept fractions, on both sides of what the grid select's
tables and the places in its lists hold.  Compared on the GPU with a sort: every index, code, scale and value, and the
residual, bit by bit."""
import pytest
import torch

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    import paper_2506_16235_b200 as nsml


def expected(vals, k, bits):
    """Indices, value section, scales (or None) and reconstructed values of the k largest |v|, ties by lower index."""
    key = vals.view(torch.int32) & 0x7FFFFFFF
    threshold = key.sort().values[key.numel() - k]
    sure = key > threshold
    ties = key == threshold
    need = k - int(sure.sum())
    tied = ties.nonzero().flatten()[:need]
    sure[tied] = True
    idx = sure.nonzero().flatten()
    v = vals[idx]
    if bits == 32:
        return idx, v.view(torch.uint8), None, v
    if bits == 16:
        half = v.to(torch.float16)
        return idx, half.view(torch.uint8), None, half.float()
    blocks = (k + 1023) // 1024
    padded = torch.zeros(blocks * 1024, device="cuda")
    padded[:k] = v.abs()
    most = padded.view(blocks, 1024).amax(1)
    scale = most / torch.full_like(most, 127.0)  # (a tensor: a scalar would be multiplied by its inverse)
    of = scale.repeat_interleave(1024)[:k]
    code = torch.where(of > 0, (v / of).round().clamp(-127, 127), torch.zeros_like(v)).to(torch.int8)
    return idx, code.view(torch.uint8), scale, code.float() * of


def check(grad, ratio, bits, mask=None, residual=None):
    n = grad.numel()
    vals = grad.float() if residual is None else grad.float() + residual
    total = vals
    if mask is not None:
        at = torch.arange(0, 32, device="cuda", dtype=torch.int32)
        pruned = ((mask[:, None] >> at) & 1).flatten()[:n].bool()
        vals = torch.where(pruned, torch.zeros_like(vals), vals)
        del pruned
    k = nsml.nsml_k_of(n, ratio)
    ws = nsml.alloc_bytes(nsml.nsml_workspace_bytes(n, nsml.NSML_BF16 if grad.dtype == torch.bfloat16 else nsml.NSML_F32), "cuda")
    if residual is None:
        payload = nsml.nsml_compress(grad, ratio, bits, prune_mask=mask, workspace=ws)
    else:
        payload = nsml.nsml_compress_feedback(grad, residual, ratio, bits, prune_mask=mask, workspace=ws)
    assert nsml.nsml_last_status(ws) == 0
    del ws
    idx, section, scale, carried = expected(vals, k, bits)
    val_off = 64 + (4 * k + 15) // 16 * 16
    assert torch.equal(payload[64:64 + 4 * k].view(torch.int32), idx.to(torch.int32)), "indices differ"
    assert torch.equal(payload[val_off:val_off + section.numel()], section), "values differ"
    if scale is not None:
        scale_off = val_off + (k + 15) // 16 * 16
        assert torch.equal(payload[scale_off:scale_off + 4 * scale.numel()].view(torch.float32), scale), "scales differ"
    if residual is not None:
        left = total.clone()
        left[idx] = torch.where(vals[idx] != 0, total[idx] - carried, total[idx])
        assert torch.equal(residual, left), "residuals differ"


def gradient(n, kind, dtype=torch.float32):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(n % 1000003)
    g = torch.randn(n, generator=gen, device="cuda")
    for i, part in enumerate(g.chunk(40)):  # tensors of different scales
        part.mul_(10.0 ** (-2.0 - (i * 7 % 5) / 2.0))
    if kind == "rows":  # an embedding table: 70 % of its rows are zero
        rows = n // 768
        g[: rows * 768].view(rows, 768)[torch.rand(rows, generator=gen, device="cuda") < 0.7] = 0.0
    if kind == "ties":
        g[torch.rand(n, generator=gen, device="cuda") < 0.5] = 0.0078125
    return g.to(dtype)


# 154,583,040 float32 elements are 255 rows of segments on 148 SMs, 310,378,496 are 512
@pytest.mark.parametrize("n", [154_583_040, 154_583_041, 200_000_007, 310_378_496, 310_378_497])
def test_float32(n):
    g = gradient(n, "plain")
    check(g, 0.5, 8)
    check(g, 0.13, 16)


@pytest.mark.parametrize("n", [155_000_001, 312_000_003])
@pytest.mark.parametrize("kind,ratio,bits", [("plain", 1.0, 16), ("plain", 0.9999, 32), ("rows", 0.5, 8), ("ties", 0.2, 8)])
def test_float32_where_little_is_left_out_or_values_repeat(n, kind, ratio, bits):
    check(gradient(n, kind), ratio, bits)


@pytest.mark.parametrize("n,ratio", [(310_378_495, 0.1), (310_378_497, 0.1), (420_000_011, 0.5), (420_000_011, 1.0)])
def test_bfloat16(n, ratio):
    check(gradient(n, "plain", torch.bfloat16), ratio, 16)


@pytest.mark.parametrize("n", [160_000_001, 311_000_033])
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
def test_residual_and_mask(n, dtype):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(7)
    mask = torch.randint(-(1 << 31), 1 << 31, ((n + 31) // 32,), generator=gen, device="cuda").to(torch.int32)
    mask &= torch.randint(-(1 << 31), 1 << 31, ((n + 31) // 32,), generator=gen, device="cuda").to(torch.int32)
    residual = torch.randn(n, generator=gen, device="cuda") * 1e-3
    g = gradient(n, "rows", dtype)
    check(g, 0.3, 8, mask=mask, residual=residual)
    check(g, 0.5, 16, mask=mask)


def test_a_large_call_leaves_nothing_behind():
    # the call after one that is near the limits of a launch
    g = gradient(154_583_041, "plain")
    nsml.nsml_compress(g, 0.5, 8)
    small = torch.randn(300_000, device="cuda")
    check(small, 0.5, 8)
    check(small, 0.01, 8)
