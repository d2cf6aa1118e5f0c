"""A call that a CUDA function refuses returns an error and leaves nothing behind: the thread's next call, which has nothing
to do with it, succeeds."""
import ctypes

import numpy as np
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    import paper_2506_16235_b200 as nsml
    from gpu_util import assert_payload_equal, oracle_compress, to_device_grad

THREAD_LOCAL = 1  # cudaStreamCaptureModeThreadLocal


def test_the_error_of_a_refused_call_does_not_reach_the_next_one():
    # waiting for the norm is refused while its stream is captured (and ends the capture)
    n = 300_000
    g = synth.config1_bucket(n=n, seed=2)
    grad, side = to_device_grad(g), torch.cuda.Stream()
    ws, norm_ws = nsml.alloc_bytes(nsml.nsml_workspace_bytes(n), "cuda"), nsml.alloc_bytes(nsml.lib.nsml_l2_workspace_bytes(), "cuda")
    payload = nsml.alloc_bytes(nsml.nsml_payload_bytes(n, 0.5, 8), "cuda")
    dense, dense_ws = torch.empty(n, device="cuda"), nsml.alloc_bytes(nsml.nsml_accumulate_workspace_bytes(n, 1), "cuda")
    weights, mask = torch.rand(n, device="cuda"), torch.zeros((n + 31) // 32, dtype=torch.int32, device="cuda")
    residual = torch.zeros(n, device="cuda")
    torch.cuda.synchronize()
    rt = ctypes.CDLL("libcudart.so.12")  # the one torch has loaded
    stream, graph, l2 = ctypes.c_void_p(side.cuda_stream), ctypes.c_void_p(), ctypes.c_double(-1.0)

    def refused():
        assert rt.cudaStreamBeginCapture(stream, THREAD_LOCAL) == 0
        rc = nsml.lib.nsml_grad_l2(grad.data_ptr(), n, nsml.NSML_F32, norm_ws.data_ptr(), norm_ws.numel(), side.cuda_stream, ctypes.byref(l2))
        assert rt.cudaStreamEndCapture(stream, ctypes.byref(graph)) != 0
        rt.cudaGetLastError()
        assert rc == nsml.NSML_ERR_CUDA and l2.value == -1.0

    calls = {
        "compress, dense": lambda: nsml.nsml_compress(grad, 0.5, 8, payload=payload, workspace=ws),
        "compress, list": lambda: nsml.nsml_compress(grad, 0.01, 8, payload=payload, workspace=ws),
        "feedback": lambda: nsml.nsml_compress_feedback(grad, residual, 0.01, 8, payload=payload, workspace=ws),
        "mask": lambda: nsml.nsml_prune_mask_build(weights, 0.01, prune_mask=mask),
        "norm": lambda: nsml.nsml_grad_l2(grad),
        "sum": lambda: nsml.nsml_decompress_accumulate([nsml.nsml_compress(grad, 0.5, 8, payload=payload, workspace=ws)], dense, workspace=dense_ws),
    }
    for name, call in calls.items():
        refused()
        call()  # raises if it fails
        torch.cuda.synchronize()
    refused()
    got = nsml.nsml_compress(grad, 0.5, 8, payload=payload, workspace=ws)
    assert nsml.nsml_last_status(ws) == 0
    assert_payload_equal(got, oracle_compress(g, 0.5, 8))
    assert nsml.nsml_grad_l2(grad) == pytest.approx(float(np.sqrt((g.astype(np.float64) ** 2).sum())), rel=1e-12)
