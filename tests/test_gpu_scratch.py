"""Scratch smaller than one launch of all rows needs.  Needs a B200."""
import pytest
import torch

from paper_2608_15531_b200 import binding as fq
from paper_2608_15531_b200 import synth

import harness as H

pytestmark = pytest.mark.gpu


def _layer(g, BN):
    K, N = 2048, 1536
    lay = synth.layer(synth.tensor_seed(15, g + BN), K, N, density=0.01, layout="mixed")
    return H.pack_layer(lay, g, BN), K


@pytest.mark.parametrize("g,BN,held", [(64, 256, 16), (64, 128, 16), (128, 256, 32), (128, 128, 32), (128, 128, 64), (64, 128, 64)])
@pytest.mark.parametrize("M", [17, 40, 128])
def test_scratch_sized_for_fewer_rows(g, BN, held, M):
    """Groups of 64 never needed more than the scratch of 16 rows, groups of 128 never more than that of 32: a caller who
    holds that much is served, in several launches.  Less is refused, and nothing is launched."""
    P, K = _layer(g, BN)
    X = synth.activations(M, M, K)
    least = 32 if g == 128 else 16
    P.ws = torch.zeros(fq.fq_workspace_bytes(P.L, min(held, M)), dtype=torch.uint8, device="cuda")
    Yref, Yabs = H.oracle_result(P, X)
    Y = H.run_fused(P, X)
    H.check_tolerances(Y, Yref, Yabs, K)
    assert (H.run_fused(P, X) == Y).all() and not P.ws[: 256 + 32768].any()
    P.ws = torch.zeros(fq.fq_workspace_bytes(P.L, min(least, M)) - 1, dtype=torch.uint8, device="cuda")
    with pytest.raises(fq.FqError) as e:
        H.run_fused(P, X)
    assert e.value.code == fq.FQ_ERR_BUFFER_TOO_SMALL


@pytest.mark.parametrize("BN", [128, 256])
@pytest.mark.parametrize("M", [17, 48, 128])
def test_the_built_in_scratch_takes_every_batch_of_a_layer_with_groups_of_64(BN, M):
    P, K = _layer(64, BN)
    X = synth.activations(M, M, K)
    Y = torch.full((M, P.L.N), 0x7fc0, dtype=torch.int16, device="cuda")
    fq.fq_fused_w4a16_outlier_gemm_noalloc(P.L, H.to_dev(X), M, *[P.d[k] for k in ("wq", "scale", "zero", "indptr", "info", "packed")], Y)
    Yref, Yabs = H.oracle_result(P, X)
    H.check_tolerances(H.bf16_bits(Y), Yref, Yabs, K)
