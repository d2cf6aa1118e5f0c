"""The line between the candidate list and the dense select: what nsml_compress_strategy says is what runs, on both sides of
every line, and both give the same payload and residual."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    import paper_2506_16235_b200 as nsml
    from gpu_util import check_compress

# (elements, kept fraction just below the line, at it) for a call by itself; for many calls in flight
LONE = [(200_001, 0.25), (3_999_999, 0.25), (4_000_000, 0.2), (11_999_999, 0.2), (12_000_000, 0.15), (39_999_999, 0.15)]
MANY = [(200_001, 0.25), (12_000_000, 0.25), (31_999_999, 0.25), (32_000_000, 0.2)]


def gradient(n, dtype):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(n)
    g = torch.randn(n, generator=gen, device="cuda")
    return (g * torch.repeat_interleave(10.0 ** (-3.0 * torch.rand(n // 4096 + 1, generator=gen, device="cuda")), 4096)[:n]).to(dtype)


def ran(g, ratio, residual):
    """The payload, the residual and whether the dense select ran."""
    left = None if residual is None else residual.clone()
    nsml.nsml_prof_reset()
    nsml.nsml_prof_enable(True)
    try:
        payload = torch.zeros(nsml.nsml_payload_bytes(g.numel(), ratio, 8), dtype=torch.uint8, device="cuda")  # (nobody writes the padding)
        if left is None:
            nsml.nsml_compress(g, ratio, 8, payload=payload)
        else:
            nsml.nsml_compress_feedback(g, left, ratio, 8, payload=payload)
        torch.cuda.synchronize()
        launches = {name: count for name, (_, count) in nsml.nsml_prof_read().items()}
    finally:
        nsml.nsml_prof_enable(False)
    assert (launches["k_select_grid"] == 1) != (launches["k_emit"] == 1)
    return payload, left, launches["k_select_grid"]


def lines(many_calls, dtype, residual):
    if many_calls:
        return MANY
    if residual:
        return LONE[:4] + [(12_000_000, 0.125), (40_000_000, 0.125)]
    return LONE + [(40_000_000, 0.1 if dtype == torch.bfloat16 else 0.125)]


@pytest.mark.parametrize("many_calls", [False, True])
@pytest.mark.parametrize("residual", [False, True])
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
def test_what_is_told_is_what_runs(dtype, residual, many_calls):
    kind = nsml.NSML_BF16 if dtype == torch.bfloat16 else nsml.NSML_F32
    for n, line in lines(many_calls, dtype, residual):
        g = gradient(n, dtype)
        start = gradient(n + 1, torch.float32)[:n].clone() if residual else None
        for ratio, dense in ((line - 2.0 / n, 0), (line, 1)):
            got = []
            for knob in (8192, 4096) if not many_calls else (4096, 8192):  # the last one is what is asked about
                nsml.nsml_set_list_block_candidates(knob)
                try:
                    told = nsml.nsml_compress_strategy(n, ratio, kind, residual)
                    got.append(ran(g, ratio, start))
                finally:
                    nsml.nsml_set_list_block_candidates(4096)
                assert got[-1][2] == told
            assert told == dense
            assert torch.equal(got[0][0], got[1][0])
            if residual:
                assert torch.equal(got[0][1].view(torch.int32), got[1][1].view(torch.int32))


def test_close_keys_need_another_histogram():
    # more keys than are exchanged within 3000 units in the last place of each other around the threshold
    n = 1_212_000
    rng = np.random.default_rng(12)
    g = (rng.standard_normal(n) * 10.0 ** rng.uniform(-6, -4, n)).astype(np.float32)
    where = rng.choice(n, 400_000, replace=False)
    g[where] = (np.float32(0.5).view(np.uint32) + rng.integers(0, 3000, where.size).astype(np.uint32)).view(np.float32)
    for ratio in (0.26, 0.32):
        check_compress(g, ratio, 16)
