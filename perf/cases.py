"""The work a data-parallel training job has libnsml do, as a list of timed cases.

A case is one call (or, for "step", one exchange step) through the Python binding, with everything a training
program keeps between steps in hand: gradients, residuals, weights, received payloads, workspaces and output
buffers, all on the GPU.  Kinds:

  compress     nsml_compress of one flat gradient bucket (float32 or bfloat16, optional pruning mask)
  feedback     nsml_compress_feedback: the same with the caller's residual (local accumulation)
  adaptive     nsml_compress_adaptive: Alg. 2 as a whole (norm, gate, mask from the weights, compress)
  accumulate   nsml_decompress_accumulate of W workers' payloads into one dense gradient
  step         one rank's exchange step over a gradient set of several buckets: every bucket is compressed and
               summed with the other workers' payloads, buckets round-robin over a few streams

Gradients take the structure real ones have: a set of tensors whose scales differ by orders of magnitude (so
that the survivors crowd into a few tensors), embedding tables of which most rows are zero, a few per cent of
heavy-tailed outliers, exact zeros; or, as the opposite extreme, one scale for the whole bucket.
"""
from __future__ import annotations

import math

import torch

import paper_2506_16235_b200 as nsml

F32, BF16 = "float32", "bfloat16"
CODECS = (8, 16, 32)
VALUE_BYTES = {8: 1, 16: 2, 32: 4}
WORKERS = (1, 2, 4, 8)
DATA = ("tensors", "outliers", "embedding", "blocks", "even")


def listed():
    return [
        # the short bucket that is left over at the end of a gradient set: launches and latency are all there is
        dict(name="compress_tail_12k", kind="compress", n=12_289, dtype=F32, ratio=0.1, bits=8, mask=False, data="tensors"),
        # one gradient vector of a megabyte-size layer (the first configuration of the benchmark)
        dict(name="compress_1M", kind="compress", n=1 << 20, dtype=F32, ratio=0.01, bits=8, mask=False, data="blocks"),
        # 25 MB buckets (PyTorch DDP's default) of a ResNet-50: a fast network lets the controller keep half of
        # the gradient; the last, shorter bucket over a slow one, where it keeps a thousandth
        dict(name="compress_25MB_half", kind="compress", n=6_553_600, dtype=F32, ratio=0.5, bits=8, mask=False, data="outliers"),
        dict(name="compress_25MB_thousandth", kind="compress", n=5_896_232, dtype=F32, ratio=0.001, bits=16, mask=False, data="outliers"),
        # a GPT-2-small gradient in 25M-element buckets; this one holds a part of the token embedding
        dict(name="compress_25M", kind="compress", n=25_000_000, dtype=F32, ratio=0.01, bits=8, mask=False, data="embedding"),
        # 64M-element bfloat16 buckets of a 1.3B-parameter decoder, sent as 16-bit values
        dict(name="compress_64M_bf16", kind="compress", n=1 << 26, dtype=BF16, ratio=0.1, bits=16, mask=False, data="tensors"),
        # the same with what sparsification leaves out carried to the next step, under a pruning mask
        dict(name="feedback_25M_masked", kind="feedback", n=25_000_000, dtype=F32, ratio=0.01, bits=8, mask=True, data="tensors"),
        # all three steps of Alg. 2 in one call; the gate fires, so 16-bit values at twice the ratio
        dict(name="adaptive_25M", kind="adaptive", n=24_439_808, dtype=F32, ratio=0.01, bits=32, gate=True, data="tensors"),
        # sums of received payloads: an odd-sized bucket added to what is there, ...
        dict(name="accumulate_1M_add", kind="accumulate", n=1_048_579, W=2, ratio=0.05, bits=16, zero_first=False, data="blocks"),
        # ... the GPT-2 bucket of four workers, ...
        dict(name="accumulate_25M_w4", kind="accumulate", n=25_000_000, W=4, ratio=0.01, bits=8, zero_first=True, data="tensors"),
        # ... and eight workers' 350M-element buckets, the largest the benchmark configurations have
        dict(name="accumulate_350M_w8", kind="accumulate", n=350_000_000, W=8, ratio=0.05, bits=8, zero_first=True, data="even"),
        # one step of one of eight ranks over a whole ResNet-50 gradient set (25 MB buckets, four streams)
        dict(name="step_resnet50", kind="step", total=25_557_032, bucket=6_553_600, W=8, ratio=0.01, bits=8, streams=4, data="outliers"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: sizes and kept fractions over their logarithms, every option that the path has."""
    kind = rng.choice(("compress", "compress", "compress", "feedback", "adaptive", "accumulate", "accumulate", "step"))
    ratio = math.exp(rng.uniform(math.log(0.001), 0.0))
    case = dict(kind=kind, ratio=ratio, bits=rng.choice(CODECS), data=rng.choice(DATA))
    if kind in ("compress", "feedback"):
        case.update(n=_log_int(rng, 4096, 1 << 26), dtype=rng.choice((F32, F32, BF16)), mask=rng.random() < 0.25)
    elif kind == "adaptive":
        case.update(n=_log_int(rng, 4096, 1 << 26), dtype=rng.choice((F32, F32, BF16)), gate=rng.random() < 0.5)
    elif kind == "accumulate":
        case.update(n=_log_int(rng, 4096, 350_000_000), W=rng.choice(WORKERS), zero_first=rng.random() < 0.75)
    else:
        buckets = rng.randint(2, 6)
        bucket = _log_int(rng, 65_536, 6_553_600)
        case.update(total=(buckets - 1) * bucket + rng.randint(1024, bucket), bucket=bucket, W=rng.choice(WORKERS),
                    streams=rng.randint(1, 4))
    # no drawn case costs more than the largest listed one
    size = "total" if kind == "step" else "n"
    while work(case)["bytes"] > (2.0e9 if kind == "accumulate" else 0.9e9):
        case[size] = case[size] // 2 + 1
    return case


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _generator(seed, salt):
    g = torch.Generator(device="cuda")
    g.manual_seed((int(seed) * 1_000_003 + salt * 7919 + 12345) % (1 << 62))
    return g


def _scales(n, gen, count, lo_exp, hi_exp):
    """Per-element scale: `count` tensors of random sizes, each with a scale log-uniform in 10**[lo, hi]."""
    cuts = torch.randint(0, n + 1, (count - 1,), generator=gen, device="cuda", dtype=torch.int64).sort().values
    ends = torch.cat([cuts, torch.tensor([n], device="cuda")])
    sizes = torch.diff(ends, prepend=torch.zeros(1, dtype=torch.int64, device="cuda"))
    scale = 10.0 ** (lo_exp + (hi_exp - lo_exp) * torch.rand(count, generator=gen, device="cuda"))
    return torch.repeat_interleave(scale, sizes, output_size=n)


def _gradient(n, data, seed, worker=0):
    """float32 gradient of n elements.  The workers of one seed share the tensors' scales (and zero rows)."""
    shared, own = _generator(seed, 0), _generator(seed, 1 + worker)
    g = torch.randn(n, generator=own, device="cuda")
    if data == "even":  # one scale: the survivors are spread evenly
        return g.mul_(1e-3)
    if data == "blocks":  # a scale per 4096 elements, 20 % exact zeros
        blocks = (n + 4095) // 4096
        scale = 10.0 ** (-4.0 + 3.0 * torch.rand(blocks, generator=shared, device="cuda"))
        g.mul_(torch.repeat_interleave(scale, 4096)[:n])
        return g.masked_fill_(torch.rand(n, generator=own, device="cuda") < 0.2, 0.0)
    if data == "outliers":  # tensors over four decades, 5 % of the values ten times as wide
        g.mul_(_scales(n, shared, max(2, min(64, n // 4096)), -5.0, -1.0))
        return torch.where(torch.rand(n, generator=own, device="cuda") < 0.05, g * 10.0, g)
    g.mul_(_scales(n, shared, max(2, min(50, n // 4096)), -4.0, -2.0))
    if data == "embedding":  # the first 60 %: a token-embedding table, 90 % of whose rows are zero
        rows = int(0.6 * n) // 768
        if rows:
            g[: rows * 768].view(rows, 768).mul_((torch.rand(rows, 1, generator=shared, device="cuda") >= 0.9).float())
    return g


def _mask(n, seed):
    """Pruning mask with about a quarter of the parameters pruned (bit set = pruned)."""
    gen = _generator(seed, 90)
    words = (n + 31) // 32
    lo, hi = -(1 << 31), 1 << 31
    a = torch.randint(lo, hi, (words,), generator=gen, device="cuda", dtype=torch.int64)
    b = torch.randint(lo, hi, (words,), generator=gen, device="cuda", dtype=torch.int64)
    return (a & b).to(torch.int32)


def _payloads(n, ratio, bits, data, seed, workers):
    """The payloads of the given workers, as they arrive from an all-gather."""
    ws = nsml.alloc_bytes(nsml.nsml_workspace_bytes(n), "cuda")
    return [nsml.nsml_compress(_gradient(n, data, seed, w), ratio, bits, workspace=ws) for w in workers]


def _bucket_sizes(case):
    return [min(case["bucket"], case["total"] - lo) for lo in range(0, case["total"], case["bucket"])]


def prepare(case, seed):
    kind, ratio, bits, data = case["kind"], case["ratio"], case["bits"], case["data"]
    state = dict(case=case)
    if kind == "accumulate":
        n, W = case["n"], case["W"]
        state["payloads"] = _payloads(n, ratio, bits, data, seed, range(W))
        state["dense"] = torch.zeros(n, device="cuda")
        state["workspace"] = nsml.alloc_bytes(nsml.nsml_accumulate_workspace_bytes(n, W), "cuda")
        return state
    if kind == "step":
        W = case["W"]
        state["streams"] = [torch.cuda.Stream() for _ in range(case["streams"])]
        largest = max(_bucket_sizes(case))
        state["workspaces"] = [(nsml.alloc_bytes(nsml.nsml_workspace_bytes(largest), "cuda"),
                                nsml.alloc_bytes(nsml.nsml_accumulate_workspace_bytes(largest, W), "cuda"))
                               for _ in state["streams"]]
        state["buckets"] = []
        for b, n in enumerate(_bucket_sizes(case)):
            state["buckets"].append(dict(
                grad=_gradient(n, data, seed + 101 * b), dense=torch.zeros(n, device="cuda"),
                payload=nsml.alloc_bytes(nsml.nsml_payload_bytes(n, ratio, bits), "cuda"),
                received=_payloads(n, ratio, bits, data, seed + 101 * b, range(1, W))))
        torch.cuda.synchronize()  # the inputs are complete before other streams read them
        return state
    n, dtype = case["n"], case["dtype"]
    grad = _gradient(n, data, seed)
    state["grad"] = grad.to(torch.bfloat16) if dtype == BF16 else grad
    code = nsml.NSML_BF16 if dtype == BF16 else nsml.NSML_F32
    if kind == "adaptive":
        gen = _generator(seed, 91)
        state["weights"] = torch.randn(n, generator=gen, device="cuda").mul_(0.02)
        state["mask"] = torch.zeros((n + 31) // 32, dtype=torch.int32, device="cuda")
        # Alg. 2's thresholds (the paper gives no values): the gate fires or not, the norm is needed either way
        state["tr_q"], state["tr_d"] = 2.0, 0.0 if case["gate"] else 1e30
        state["payload"] = nsml.alloc_bytes(nsml.lib.nsml_adaptive_payload_bytes(n, ratio, state["tr_q"], bits), "cuda")
        state["workspace"] = nsml.alloc_bytes(nsml.lib.nsml_adaptive_workspace_bytes(n, code), "cuda")
        return state
    state["mask"] = _mask(n, seed) if case["mask"] else None
    state["payload"] = nsml.alloc_bytes(nsml.nsml_payload_bytes(n, ratio, bits), "cuda")
    state["workspace"] = nsml.alloc_bytes(nsml.nsml_workspace_bytes(n, code), "cuda")
    if kind == "feedback":
        state["residual"] = torch.zeros(n, device="cuda")
    return state


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------
def _step(state):
    case, streams = state["case"], state["streams"]
    current = torch.cuda.current_stream()
    for s in streams:
        s.wait_stream(current)
    for b, bucket in enumerate(state["buckets"]):
        s = streams[b % len(streams)]
        ws, aws = state["workspaces"][b % len(streams)]
        own = nsml.nsml_compress(bucket["grad"], case["ratio"], case["bits"], payload=bucket["payload"], workspace=ws, stream=s)
        nsml.nsml_decompress_accumulate([own] + bucket["received"], bucket["dense"], workspace=aws, stream=s, sized=True)
        bucket["own"] = own
    for s in streams:
        current.wait_stream(s)
    return {"own": [b["own"] for b in state["buckets"]], "dense": [b["dense"] for b in state["buckets"]]}


def run(state):
    case = state["case"]
    kind, ratio, bits = case["kind"], case["ratio"], case["bits"]
    if kind == "step":
        return _step(state)
    if kind == "accumulate":
        return nsml.nsml_decompress_accumulate(state["payloads"], state["dense"], zero_first=case["zero_first"],
                                               workspace=state["workspace"])
    if kind == "compress":
        return nsml.nsml_compress(state["grad"], ratio, bits, prune_mask=state["mask"], payload=state["payload"],
                                  workspace=state["workspace"])
    if kind == "feedback":
        payload = nsml.nsml_compress_feedback(state["grad"], state["residual"], ratio, bits, prune_mask=state["mask"],
                                              payload=state["payload"], workspace=state["workspace"])
        return {"payload": payload, "residual": state["residual"]}
    payload, used_ratio, used_bits, l2, mask = nsml.nsml_compress_adaptive(
        state["grad"], ratio, state["tr_q"], state["tr_d"], bits, weights=state["weights"], prune_mask=state["mask"],
        payload=state["payload"], workspace=state["workspace"])
    return {"payload": payload, "ratio": used_ratio, "bits": used_bits, "l2": l2, "mask": mask}


# ---------------------------------------------------------------------------
# what a pass cannot do without, and how close results have to be
# ---------------------------------------------------------------------------
def _payload_bytes(n, ratio, bits):
    k = min(n, max(1, math.ceil(ratio * n)))
    return k * (4 + VALUE_BYTES[bits]) + (k / 256 if bits == 8 else 0)


def work(case):
    """Bytes of the inputs read once and the outputs written once; operations: a compare per element (a square
    and an add for the norm, an add for the residual), a multiply and an add per payload entry summed."""
    kind, ratio, bits = case["kind"], case["ratio"], case["bits"]
    if kind == "accumulate":
        n, W = case["n"], case["W"]
        entries = W * max(1.0, ratio * n)
        return {"bytes": W * _payload_bytes(n, ratio, bits) + (4 if case["zero_first"] else 8) * n, "flops": 2 * entries}
    if kind == "step":
        moved = flops = 0.0
        for n in _bucket_sizes(case):
            moved += 4 * n + case["W"] * _payload_bytes(n, ratio, bits) + 4 * n
            flops += n + 2 * case["W"] * ratio * n
        return {"bytes": moved, "flops": flops}
    n = case["n"]
    element = 2 if case["dtype"] == BF16 else 4
    if kind == "adaptive":
        used_ratio, used_bits = (min(1.0, 2 * ratio), 16) if case["gate"] else (ratio, bits)
        return {"bytes": element * n + 4 * n + n / 8 + _payload_bytes(n, used_ratio, used_bits), "flops": 4 * n}
    moved = element * n + _payload_bytes(n, ratio, bits) + (n / 8 if case["mask"] else 0)
    if kind == "feedback":
        return {"bytes": moved + 8 * n, "flops": 2 * n}
    return {"bytes": moved, "flops": n}


def tolerance(case):
    """Payloads, masks and residual arithmetic are defined to the bit (bytes are compared whole); sums of W
    float32 values and the norm may differ by the order of the additions."""
    if case["kind"] == "compress":
        return "exact"
    return {"rel": 1e-6, "max": 1e-5}
