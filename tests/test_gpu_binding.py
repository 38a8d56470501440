"""The binding of the fused calls on tensors that share storage until they are written, and on sparse ones.  Needs a B200."""
import pytest
import torch

from paper_2608_15531_b200 import binding as fq
from paper_2608_15531_b200 import synth

import harness as H

pytestmark = pytest.mark.gpu


def _weights(P):
    return [P.d[k] for k in ("wq", "scale", "zero", "indptr", "info", "packed")]


def test_a_lazy_clone_that_is_written_leaves_its_source_alone():
    """Y, the scratch and the staging buffers as copy-on-write clones: the call writes into storage of their own."""
    K, N, M = 2048, 1536, 8
    P = H.pack_layer(synth.layer(synth.tensor_seed(16, 1), K, N, density=0.01, layout="mixed"), 128)
    X = synth.activations(1, M, K)
    want = torch.from_numpy(H.run_fused(P, X).view("int16"))
    ys, xs, ws = torch.full((M, N), 7, dtype=torch.int16, device="cuda"), torch.full((M, K), 9, dtype=torch.int16, device="cuda"), torch.zeros_like(P.ws)
    y, x, scratch = torch._lazy_clone(ys), torch._lazy_clone(xs), torch._lazy_clone(ws)
    fq.fq_fused_w4a16_outlier_gemm(P.L, H.to_dev(X), M, *_weights(P), y, scratch)
    assert torch.equal(y.cpu(), want) and bool((ys == 7).all()) and not ws.any()
    y = torch._lazy_clone(ys)
    Xh, Yh = torch.from_numpy(X.view("int16")).pin_memory(), torch.zeros((M, N), dtype=torch.int16).pin_memory()
    fq.fq_fused_host_io(P.L, Xh, M, x, *_weights(P), y, Yh, P.ws)
    assert torch.equal(Yh, want) and bool((ys == 7).all()) and bool((xs == 9).all())


def test_a_sparse_tensor_is_refused():
    P = H.pack_layer(synth.layer(synth.tensor_seed(16, 2), 256, 256, density=0.0), 128)
    for X in (torch.eye(4, device="cuda").to_sparse(), torch.eye(4, device="cuda").to_sparse_csr()):
        with pytest.raises((ValueError, RuntimeError)):
            fq.fq_fused_w4a16_outlier_gemm(P.L, X, 1, *_weights(P), torch.empty((1, 256), dtype=torch.int16, device="cuda"), P.ws)
