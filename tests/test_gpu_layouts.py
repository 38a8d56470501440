"""Layouts that say little of their arrays, or what is not so: through every kernel that serves them.  Needs a B200."""
import numpy as np
import pytest

from paper_2608_15531_b200 import binding as fq
from paper_2608_15531_b200 import synth

import harness as H

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("K,N,g,BN", [(2944, 1408, 128, 128), (1024, 1024, 64, 256)])
@pytest.mark.parametrize("M", [16, 17, 48, 128])
def test_the_dense_half_is_the_fused_kernel_without_outliers(K, N, g, BN, M):
    """fq_unfused_gemm on a layer with outliers (no sparse array is given), against the oracle's dense half; and bit for bit the fused
    call on the same codes without outliers."""
    P = H.pack_layer(synth.layer(synth.tensor_seed(14, 9), K, N, density=0.01, layout="mixed"), g, BN)
    X = synth.activations(2, M, K)
    Y = H.run_unfused(P, X, with_spmm=False)
    Yref, Yabs = H.oracle_result(P, X, dense_only=True)
    H.check_tolerances(Y, Yref, Yabs, K)
    E = H.pack_layer(synth.layer(synth.tensor_seed(14, 9), K, N, density=0.0), g, BN)
    E.d |= {k: P.d[k] for k in ("wq", "scale", "zero")}
    assert np.array_equal(H.run_fused(E, X), Y)


def _repeated_layer(seed, K, N, g, density=0.01):
    lay = synth.layer(synth.tensor_seed(14, seed), K, N, density=density, layout="uniform")
    lay.coo_k, lay.coo_n, lay.coo_v = (np.concatenate([a, a[:50]]) for a in (lay.coo_k, lay.coo_n, lay.coo_v))
    return H.pack_layer(lay, g)


@pytest.mark.parametrize("M", [9, 16, 24, 40, 128])
def test_a_saved_layout_that_says_nothing_of_repeats(M):
    """A layout struct as encoders wrote it before repeated positions were told apart (the three maxima and tilecoo_encoded = 1,
    whether positions repeat or not), saved and loaded again: the sum of the outliers of a position counts."""
    K, N = 4096, 2048
    P = _repeated_layer(1, K, N, 128)
    assert P.L.tilecoo_encoded == 2
    P.L.abi, P.L.tilecoo_encoded = 2, 1
    P.L = fq.Layout.from_buffer_copy(bytes(P.L))
    X = synth.activations(3, M, K)
    cols = np.unique(P.layer.coo_n[-50:])
    Yref, Yabs = H.oracle_result(P, X, cols=cols)
    H.check_tolerances(H.run_fused(P, X)[:, cols], Yref, Yabs, K)


@pytest.mark.parametrize("K,N", [(1024, 768), (2048, 6144)])
@pytest.mark.parametrize("M", [1, 8, 16, 17])
@pytest.mark.parametrize("streaming_only", [False, True])
def test_a_layout_without_outliers_on_arrays_that_have_some(K, N, M, streaming_only):
    """The struct of a layer without outliers with the arrays of one that has some: reported, by every kernel, as the
    descriptors that reach past their tile are; the same struct with its own (empty) arrays is not."""
    P = H.pack_layer(synth.layer(synth.tensor_seed(14, 5), K, N, density=0.03, layout="uniform"), 128)
    E = H.pack_layer(synth.layer(synth.tensor_seed(14, 6), K, N, density=0.0), 128)
    assert E.L.max_tile_packets == 0 and E.L.tilecoo_encoded == 1
    X = synth.activations(4, M, K)
    H.run_fused(E, X, streaming_only=streaming_only)
    mine, E.d = E.d, P.d
    with pytest.raises(fq.FqError) as e:
        H.run_fused(E, X, streaming_only=streaming_only)
    assert e.value.code == fq.FQ_ERR_FORMAT
    E.d = mine
    cols = np.arange(0, N, 37, dtype=np.uint32)
    Yref, Yabs = H.oracle_result(E, X, cols=cols)
    H.check_tolerances(H.run_fused(E, X, streaming_only=streaming_only)[:, cols], Yref, Yabs, K)
