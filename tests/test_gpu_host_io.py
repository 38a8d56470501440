"""Calls from host memory to host memory: every kind of copy, and staging buffers that are used again at once.  Needs a B200."""
import mmap

import numpy as np
import pytest
import torch

from paper_2608_15531_b200 import binding as fq
from paper_2608_15531_b200 import synth

import harness as H

pytestmark = pytest.mark.gpu


def _weights(P):
    return [P.d[k] for k in ("wq", "scale", "zero", "indptr", "info", "packed")]


@pytest.mark.parametrize("M", [1, 4, 8, 16, 24])
@pytest.mark.parametrize("streaming_only", [False, True])
def test_staging_buffers_used_again_at_once(M, streaming_only):
    """Calls that follow each other on one stream share x_dev, y_dev and the scratch and differ in X: each call's kernels are
    resident while the call before is still writing what they read.  Every result, bit for bit, against the call on a copy of
    its own in device memory."""
    K, N = 2048, 2304
    P = H.pack_layer(synth.layer(synth.tensor_seed(13, 1), K, N, density=0.01, layout="mixed"), 128)
    P.L.kernel_hint = 1 if streaming_only else 0
    calls = 12
    Xh = [torch.from_numpy(synth.activations(100 + i, M, K).view(np.int16)).pin_memory() for i in range(calls)]
    Yh = [torch.zeros((M, N), dtype=torch.int16).pin_memory() for _ in range(calls)]
    x, y = torch.empty((M, K), dtype=torch.int16, device="cuda"), torch.empty((M, N), dtype=torch.int16, device="cuda")
    for rep in range(3):
        for Xi, Yi in zip(Xh, Yh):
            fq.fq_fused_host_io_async(P.L, Xi, M, x, *_weights(P), y, Yi, P.ws)
        torch.cuda.synchronize()
        for Xi, Yi in zip(Xh, Yh):
            Y = torch.empty((M, N), dtype=torch.int16, device="cuda")
            fq.fq_fused_w4a16_outlier_gemm(P.L, Xi.cuda(), M, *_weights(P), Y, P.ws)
            assert torch.equal(Y.cpu(), Yi)
            Yi.zero_()


@pytest.mark.parametrize("K,N,M", [(1024, 768, 8), (16512, 256, 128), (256, 16640, 128)])
def test_every_kind_of_host_memory(K, N, M):
    """Pinned, pinned at an address that is no multiple of 16, pageable (tensor and numpy array); short, and X or Y longer than what a
    kernel copies (4 MB)."""
    P = H.pack_layer(synth.layer(synth.tensor_seed(13, K % 97), K, N, density=0.01, layout="uniform"), 128)
    Xb = synth.activations(5, M, K)
    Y = H.run_fused(P, Xb)
    x, y = torch.empty((M, K), dtype=torch.int16, device="cuda"), torch.empty((M, N), dtype=torch.int16, device="cuda")

    def pinned(rows, cols, shift):
        return torch.zeros(rows * cols + shift, dtype=torch.int16).pin_memory()[shift:].view(rows, cols)

    for Xh, Yh in ((pinned(M, K, 0), pinned(M, N, 0)), (pinned(M, K, 1), pinned(M, N, 3)), (pinned(M, K, 0), torch.zeros((M, N), dtype=torch.int16)),
                   (torch.zeros((M, K), dtype=torch.int16), pinned(M, N, 0)), (np.zeros((M, K), dtype=np.int16), np.zeros((M, N), dtype=np.int16))):
        Xh[:] = torch.from_numpy(Xb.view(np.int16)) if torch.is_tensor(Xh) else Xb.view(np.int16)
        fq.fq_fused_host_io(P.L, Xh, M, x, *_weights(P), y, Yh, P.ws)
        assert np.array_equal(np.asarray(Yh).view(np.uint16), Y)
        x.zero_(), y.zero_()


@pytest.mark.parametrize("side", ["X", "Y"])
def test_host_memory_that_is_pinned_in_part(side):
    """Only the first 4 KB of a buffer are registered: no kernel may copy it.  The copy engine's copy refuses it or copies it, and
    a result that is returned is right."""
    K, N, M = 1024, 1024, 8
    P = H.pack_layer(synth.layer(synth.tensor_seed(13, 7), K, N, density=0.01, layout="uniform"), 128)
    Xb = synth.activations(6, M, K)
    Y = H.run_fused(P, Xb)
    Xh, Yh = torch.from_numpy(Xb.view(np.int16).copy()).pin_memory(), torch.zeros((M, N), dtype=torch.int16).pin_memory()
    pages = np.frombuffer(mmap.mmap(-1, 1 << 16), dtype=np.int16)
    part = torch.from_numpy(pages[: M * K]).view(M, K)
    if side == "X":
        part.copy_(Xh)
        Xh = part
    else:
        Yh = part
    cudart = torch.cuda.cudart()
    assert int(cudart.cudaHostRegister(part.data_ptr(), 4096, 0)) == 0
    try:
        x, y = torch.empty((M, K), dtype=torch.int16, device="cuda"), torch.empty((M, N), dtype=torch.int16, device="cuda")
        try:
            fq.fq_fused_host_io(P.L, Xh, M, x, *_weights(P), y, Yh, P.ws)
            assert np.array_equal(Yh.numpy().view(np.uint16), Y)
        except fq.FqError as e:
            assert e.code == fq.FQ_ERR_CUDA and "copy of " + side in str(e)
        torch.cuda.synchronize()
    finally:
        assert int(cudart.cudaHostUnregister(part.data_ptr())) == 0
    assert np.array_equal(H.run_fused(P, Xb), Y)


@pytest.mark.parametrize("M", [1, 8, 40])
def test_a_captured_call_reads_its_buffers_anew(M):
    """A call from pinned to pinned memory in a CUDA graph, replayed with other values in the same buffers."""
    K, N = 2048, 2304
    P = H.pack_layer(synth.layer(synth.tensor_seed(13, 1), K, N, density=0.01, layout="mixed"), 128)
    Xh, Yh = torch.zeros((M, K), dtype=torch.int16).pin_memory(), torch.zeros((M, N), dtype=torch.int16).pin_memory()
    x, y = torch.empty((M, K), dtype=torch.int16, device="cuda"), torch.empty((M, N), dtype=torch.int16, device="cuda")
    fq.fq_fused_host_io(P.L, Xh, M, x, *_weights(P), y, Yh, P.ws)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        fq.fq_fused_host_io_async(P.L, Xh, M, x, *_weights(P), y, Yh, P.ws)
    for i in range(3):
        Xb = synth.activations(200 + i, M, K)
        Xh.copy_(torch.from_numpy(Xb.view(np.int16)))
        graph.replay()
        torch.cuda.synchronize()
        assert np.array_equal(Yh.numpy().view(np.uint16), H.run_fused(P, Xb))
