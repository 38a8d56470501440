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


def _set_outliers(lay, mask, seed):
    rng = np.random.default_rng(seed)
    kk, nn = np.nonzero(mask)
    vb = ((rng.uniform(0.12, 0.4, size=kk.size) * rng.choice([-1, 1], size=kk.size)).astype(np.float32).view(np.uint32) >> 16).astype(np.uint16)
    lay.mask, lay.coo_k, lay.coo_n, lay.coo_v = mask, kk.astype(np.uint32), nn.astype(np.uint32), vb
    lay.W[kk, nn] = synth.bf16_bits_to_f32(vb)
    return lay


def _tails(K, N, oversized):
    """Columns of 17 to 100 outliers in a tile, several of them in one strip and one bucket, on 1 % of noise; or a tile that is all
    outliers (8192 packets, more than a stage holds) beside a hot row and a hot column."""
    lay = synth.layer(synth.tensor_seed(14, 20 + oversized), K, N, density=0.0 if oversized else 0.01, layout="uniform")
    mask = lay.mask.copy()
    rng = np.random.default_rng(4)
    if oversized:
        mask[128:256, 0:256] = 1
        mask[3, 256:512] = 1
        mask[0:128, 400] = 1
    else:
        for col, cnt in ((3, 100), (12, 40), (27, 17), (5, 32)):
            mask[0:128, col] = 0
            mask[rng.choice(128, size=cnt, replace=False), col] = 1
        mask[256 + rng.choice(128, size=77, replace=False), 256 + 130] = 1
    return _set_outliers(lay, mask, 5)


@pytest.mark.parametrize("encoding", ["unknown", "repeated"])
@pytest.mark.parametrize("oversized", [False, True])
@pytest.mark.parametrize("g", [64, 128])
@pytest.mark.parametrize("M", [1, 4, 8, 16, 40])
def test_tails_and_oversized_tiles_of_encodings_that_the_tcgen05_kernel_does_not_serve(encoding, oversized, g, M):
    """The general forms of the streaming kernel (one and two octets of rows) and the short-job kernel's walk over tails."""
    K, N = 512, 512
    lay = _tails(K, N, oversized)
    if encoding == "repeated":
        lay.coo_k, lay.coo_n, lay.coo_v = (np.concatenate([a, a[::200]]) for a in (lay.coo_k, lay.coo_n, lay.coo_v))
    P = H.pack_layer(lay, g, 256)
    assert P.L.max_tail_packets > 0 and P.L.tilecoo_encoded == (2 if encoding == "repeated" else 1)
    if encoding == "unknown":
        P.L.max_tile_packets = P.L.max_bucket_packets = P.L.max_tail_packets = P.L.tilecoo_encoded = 0
    X = synth.activations(7, M, K)
    Yref, Yabs = H.oracle_result(P, X)
    for streaming_only in (False, True):
        H.check_tolerances(H.run_fused(P, X, streaming_only=streaming_only), Yref, Yabs, K)


@pytest.mark.parametrize("BN,density,layout", [(256, 0.02, "mixed"), (128, 0.02, "clustered"), (256, 0.05, "clustered")])
@pytest.mark.parametrize("g", [64, 128])
@pytest.mark.parametrize("M", [9, 24, 48, 64, 100, 128])
def test_fp16_outliers_in_two_parts_on_every_variant_of_the_tcgen05_kernel(BN, density, layout, g, M):
    """IEEE binary16 values with all ten fraction bits in use, columns with and without tails; several units to a CTA and an
    odd number of k-steps, so that each scatter group's tiles are written, read and cleared in turn for both parts."""
    K, N = 4480, 2048
    lay = synth.layer(synth.tensor_seed(14, 30 + BN), K, N, density=density, layout=layout)
    rng = np.random.default_rng(8)
    vals = (rng.uniform(0.12, 0.4, size=lay.coo_k.size) * rng.choice([-1, 1], size=lay.coo_k.size)).astype(np.float16)
    lay.coo_v = vals.view(np.uint16).copy()
    lay.W[lay.coo_k, lay.coo_n] = vals.astype(np.float32)
    P = H.pack_layer(lay, g, BN, value_type=fq.FQ_VALUE_FP16)
    assert (P.L.max_tail_packets > 0) == (layout == "clustered")
    X = synth.activations(9, M, K)
    cols = np.unique(np.concatenate([np.arange(0, N, 53), np.argsort(lay.mask.sum(axis=0))[::-1][:8]])).astype(np.uint32)
    Yref, Yabs = H.oracle_result(P, X, cols=cols)
    Y = H.run_fused(P, X)
    H.check_tolerances(Y[:, cols], Yref, Yabs, K)
    assert np.array_equal(H.run_fused(P, X), Y)


@pytest.mark.parametrize("M", [48, 128])
@pytest.mark.parametrize("g", [64, 128])
def test_fp16_outliers_keep_their_ten_fraction_bits_in_larger_launches(g, M):
    """1 + 2^-9 and -1 in one column, activations 512 in both rows, nothing else: Y is exactly 1 (0 without the second part)."""
    K, N = 256, 512
    lay = synth.layer(1, K, N, density=0.0)
    lay.W[:] = 0.0
    rows, cols = np.array([3, 200, 77, 130], dtype=np.uint32), np.array([5, 5, 300, 300], dtype=np.uint32)
    vals = np.array([1 + 2.0 ** -9, -1.0, -(1 + 2.0 ** -10), 1.0], dtype=np.float16)
    lay.mask = np.zeros((K, N), dtype=np.uint8)
    lay.mask[rows, cols] = 1
    lay.coo_k, lay.coo_n, lay.coo_v = rows, cols, vals.view(np.uint16).copy()
    lay.W[rows, cols] = vals.astype(np.float32)
    P = H.pack_layer(lay, g, value_type=fq.FQ_VALUE_FP16)
    X = np.zeros((M, K), dtype=np.uint16)
    X[:, rows] = 0x4400                                       # 512.0
    Y = H.bits_to_f64(H.run_fused(P, X))
    assert np.all(Y[:, 5] == 1.0) and np.all(Y[:, 300] == -0.5)
    Y[:, [5, 300]] = 0
    assert not Y.any()
