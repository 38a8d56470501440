"""Either side of the rules that choose a launch's kernel, on sampled columns against the oracle.  Needs a B200."""
import dataclasses

import numpy as np
import pytest
import torch

from paper_2608_15531_b200 import synth

import harness as H

pytestmark = pytest.mark.gpu

_SHAPES = [
    (2048, 4096, 0.01, (9, 16)),           # 16 k-steps, shallow buckets: a short job; deep ones: tcgen05
    (2048, 4096, 0.05, (9, 16)),
    (2176, 4096, 0.01, (9, 16)),           # 17 k-steps: tcgen05
    (1024, 16512, 0.01, (2, 8)),           # tiles of 128 columns, one group of dense warps: tcgen05
    (8192, 6272, 0.01, (4, 5)),            # 3136 units: tcgen05 from five rows up
    (8192, 8320, 0.01, (1, 2, 4)),         # 4160 units: from two rows up, unless buckets are deep
    (8192, 8320, 0.05, (2, 5)),
    (2048, 3072, 0.01, (1, 4)),            # both builds of the short-job kernel: 96 strips, 97 and more
    (2048, 3200, 0.01, (1, 4)),
    (2048, 2048, 0.01, (5, 8)),            # and 16 k-steps, 17 and more
    (2176, 2048, 0.01, (5, 8)),
    (6016, 4096, 0.01, (5, 8)),
    (2304, 7296, 0.01, (4, 5)),            # tiles of 128 columns, a second group of dense warps only by a split along the tiles: streaming;
    (2304, 7296, 0.05, (4, 5)),            # from five rows up, if buckets are deep, tcgen05
    (2048, 12800, 0.01, (1, 8)),           # streaming kernel, tiles for two units more: they bring the second group
    (1664, 14336, 0.01, (4, 8)),           # one group either way: ranges with outliers and five rows or more, else tiles
    (1664, 14336, 0.0, (1, 16)),
    (8192, 6400, 0.01, (4, 5)),            # five CTAs to a tile up to four rows, ranges beyond
    (3840, 15360, 0.01, (1, 5)),           # two, 15 units
    (5120, 16384, 0.01, (1,)),             # two, 20 units: ranges, without outliers tiles
    (5120, 16384, 0.0, (1, 5)),
    (6272, 8832, 0.0, (1, 8)),             # tiles of 128 columns and a grid of fewer CTAs than SMs, ranges
    (6528, 5504, 0.01, (1, 2)),
]


@pytest.mark.parametrize("K,N,density,rows", _SHAPES)
@pytest.mark.parametrize("g", [64, 128])
def test_either_side_of_a_rule(K, N, density, rows, g):
    lay = synth.layer(synth.tensor_seed(17, K // 128 + N // 128), K, N, density=density, layout="uniform")
    P = H.pack_layer(lay, g)
    cols = np.unique(np.concatenate([np.arange(0, N, 97), [N - 1]])).astype(np.uint32)
    for M in rows:
        X = synth.activations(lay.seed + M, M, K)
        Y = H.run_fused(P, X)
        Yref, Yabs = H.oracle_result(P, X, cols=cols)
        H.check_tolerances(Y[:, cols], Yref, Yabs, K)
        assert np.array_equal(H.run_fused(P, X), Y)


# Layers whose column tiles are shared by several CTAs of the tcgen05 kernel.  On 148 SMs: splits along the tiles 8192 x 1024 (18 CTAs to a
# tile), 2944 x 1152 (16), 4096 x 4096 (4), 3072 x 5120 (3) and 1536 x 9472 (2); contiguous ranges, in which a CTA has parts of two tiles,
# 5120 x 5120 (11 of a tile's 40 units; at 33 to 64 rows and groups of 128 a split, three to a tile), 14336 x 4096 (25 of 112; a split, four) and
# 2944 x 11136 (14 of 23); test_shares.py holds these plans.  Up to 32 rows the whole CTA does the sums at the end of its range, and the
# first tile's too with 17 to 32, or with groups of 64; beyond, either the CTA or the drain warps, by rows and contributors (tc_coop).
# Rows at the edges of the sets of 32 rows, of the quads of rows that a thread takes, and of its second and third pass.
@pytest.mark.parametrize("K,N", [(8192, 1024), (2944, 1152), (4096, 4096), (3072, 5120), (1536, 9472), (5120, 5120), (14336, 4096), (2944, 11136)])
@pytest.mark.parametrize("g", [64, 128])
def test_tiles_with_many_contributors(K, N, g):
    lay = synth.layer(synth.tensor_seed(18, K // 128 + N // 128), K, N, density=0.01, layout="mixed")
    P = H.pack_layer(lay, g)
    cols = np.unique(np.concatenate([np.arange(0, N, 61), [N - 1]])).astype(np.uint32)
    X = synth.activations(lay.seed, 128, K)
    Yref, Yabs = H.oracle_result(P, X, cols=cols)
    for M in (9, 16, 17, 31, 32, 33, 48, 56, 57, 63, 65, 100, 128):
        Y = H.run_fused(P, X[:M])
        H.check_tolerances(Y[:, cols], Yref[:M], Yabs[:M], K)
        for _ in range(3):
            assert np.array_equal(H.run_fused(P, X[:M]), Y)


def _layer_with_slow_units(K, N, ctas):
    """A layer for contiguous ranges of `ctas` CTAs, and the column tiles of 128 that its slow units are in: the first units of ranges that begin
    inside a tile and end in the next are half outliers, whose scattering takes many times as long as all that the tile's other CTAs
    have to do.  So those CTAs, seldom the last to be done with their first tile, are the last."""
    KT, NT = K // 128, N // 128
    q, r = divmod(NT * KT, ctas)
    begins = [c * q + min(c, r) for c in range(ctas + 1)]
    across = [c for c in range(ctas) if begins[c] % KT and begins[c] // KT != (begins[c + 1] - 1) // KT]
    lay = synth.layer(synth.tensor_seed(19, KT + NT), K, N, density=0.01, layout="uniform")
    rng = np.random.default_rng(KT * NT)
    V = np.zeros((K, N), dtype=np.uint16)
    V[lay.coo_k, lay.coo_n] = lay.coo_v
    tiles = []
    for c in across[::len(across) // 5]:
        tn, kt = divmod(begins[c], KT)
        block = np.s_[kt * 128:(kt + 1) * 128, tn * 128:(tn + 1) * 128]
        bits = (synth.SIGMA * rng.uniform(6, 20, (128, 128)) * rng.choice([-1, 1], (128, 128))).astype(np.float32).view(np.uint32) >> 16
        new = (rng.random((128, 128)) < 0.5) & (lay.mask[block] == 0)
        V[block][new] = bits[new]
        lay.mask[block][new] = 1
        tiles.append(tn)
    k, n = np.nonzero(lay.mask)
    lay.W[k, n] = synth.bf16_bits_to_f32(V[k, n])
    return dataclasses.replace(lay, coo_k=k.astype(np.uint32), coo_n=n.astype(np.uint32), coo_v=V[k, n]), tiles


@pytest.mark.parametrize("K,N", [(5120, 5120), (2944, 11136)])
@pytest.mark.parametrize("g", [64, 128])
def test_a_range_that_is_the_last_to_finish_its_first_tile(K, N, g):
    """Ranges of 11 and 14 units of tiles of 40 and 23 (but of 5120 x 5120, at one row and at 33 to 64 with groups of 128, a split along the tiles)."""
    lay, tiles = _layer_with_slow_units(K, N, min(torch.cuda.get_device_properties(0).multi_processor_count, 192))
    P = H.pack_layer(lay, g)
    cols = np.unique(np.concatenate([np.arange(0, N, 61)] + [np.arange(t * 128, t * 128 + 128) for t in tiles])).astype(np.uint32)
    X = synth.activations(lay.seed, 128, K)
    Yref, Yabs = H.oracle_result(P, X, cols=cols)
    for M in (1, 9, 16, 17, 30, 32, 48, 64, 96, 128):
        Y = H.run_fused(P, X[:M])
        H.check_tolerances(Y[:, cols], Yref[:M], Yabs[:M], K)
        assert np.array_equal(H.run_fused(P, X[:M]), Y)
