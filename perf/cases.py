"""What is timed: the fused W4A16 + outlier matmul as a decoder uses it, call by call and projection by projection,
from one row to the 128 rows that a call takes, and the packing of a matrix that comes before.

Three kinds of case:
  linear  one fused call on one K x N layer
  block   the four linear layers of one decoder block (the LLaMA-3-8B shapes this repository is tuned and benchmarked
          on), one fused call each, one after the other on the stream
  pack    quantising, packing and encoding one K x N matrix on the host
With "host" a linear or block case takes its activations from pinned host memory and brings its results back there.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2608_15531_b200 import binding as fq
from paper_2608_15531_b200 import synth

BLOCK = [(K, N) for _, K, N in synth.LLAMA3_8B]
MAX_WEIGHTS = 8192 * 57344            # the largest listed layer
MAX_ROW_WEIGHTS = 128 * sum(K * N for K, N in BLOCK)      # rows x weights of the listed case with the most operations


def _linear(name, K, N, M, group=128, density=0.01, layout="mixed", host=False):
    return dict(name=name, kind="linear", K=K, N=N, M=M, group=group, density=density, layout=layout, host=host)


def _block(name, M, host=False):
    return dict(name=name, kind="block", K=0, N=0, M=M, group=128, density=0.01, layout="mixed", host=host)


def listed():
    return [
        # the smallest call: one token through the smallest projection of the 8B decoder (latency and launch cost)
        _linear("o_proj m1", 4096, 4096, 1),
        # one token through a decoder block: the ordinary decode step of a single user
        _block("block m1", 1),
        # small and full decode batches through a block
        _block("block m8", 8),
        _block("block m16", 16),
        # more users at once, up to the largest batch a call takes (also a short prefill or a speculative draft)
        _block("block m32", 32),
        _block("block m128", 128),
        # the largest matrix (70B gate_up), a few rows
        _linear("70b gate_up m4", 8192, 57344, 4),
        # finer groups on the shape of the batch sweep, in the middle of the batch range
        _linear("g64 m64", 8192, 28672, 64, group=64),
        # ragged: an odd number of rows, row tiles and column tiles, a width that is no multiple of 256
        _linear("ragged m5", 2944, 11136, 5, group=64, density=0.005, layout="uniform"),
        # a trained model's hot channels: outliers crowded into few rows and columns
        _linear("hot m8", 4096, 14336, 8, density=0.02, layout="clustered"),
        # activations from the host, results to the host: what a caller outside the GPU's stream pays for a step
        _block("block m8 host", 8, host=True),
        # the offline step every matrix goes through once: quantise, pack, encode
        dict(name="pack", kind="pack", K=4096, N=4096, M=0, group=128, density=0.01, layout="mixed", host=True),
    ]


def _log_uniform(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _option(rng):
    """A density and a layout that go together (hot rows hold at most three quarters of their weights as outliers)."""
    layout = rng.choice(["mixed", "mixed", "uniform", "clustered"])
    density = rng.choice([0.005, 0.01, 0.01] if layout == "mixed" else [0.0, 0.005, 0.01, 0.02, 0.03, 0.05] if layout == "uniform"
                         else [0.01, 0.02])
    return density, layout


def draw(rng):
    u = rng.random()
    if u < 0.08:
        K, N = (128 * round(_log_uniform(rng, 8, 64)) for _ in range(2))
        density, layout = _option(rng)
        return dict(kind="pack", K=K, N=N, M=0, group=rng.choice([64, 128, 128]), density=density, layout=layout, host=True)
    M = min(128, round(_log_uniform(rng, 1, 128)))
    if u < 0.25:
        density, layout = _option(rng)
        return dict(kind="block", K=0, N=0, M=M, group=rng.choice([64, 128, 128]), density=density, layout=layout,
                    host=rng.random() < 0.2)
    while True:
        K, N = 128 * round(_log_uniform(rng, 8, 224)), 128 * round(_log_uniform(rng, 8, 448))
        if K * N <= MAX_WEIGHTS and M * K * N <= MAX_ROW_WEIGHTS:
            break
    density, layout = _option(rng)
    return dict(kind="linear", K=K, N=N, M=M, group=rng.choice([64, 128, 128]), density=density, layout=layout,
                host=rng.random() < 0.1)


# ------------------------------------------------------------------------------------------------------- inputs

def _outlier_positions(gen, K, N, density, layout):
    """(k, n) of the outliers, on the GPU.  uniform: everywhere alike; mixed: half of them in 1 % of the rows;
    clustered: 80 % of them in 0.5 % of the rows and 0.5 % of the columns, which are filled to three quarters at most."""
    if density == 0.0:
        return torch.empty(0, dtype=torch.int64, device="cuda"), torch.empty(0, dtype=torch.int64, device="cuda")
    p = torch.empty(K, N, device="cuda")
    if layout == "uniform":
        p.fill_(density)
    elif layout == "mixed":
        rows = torch.randperm(K, generator=gen, device="cuda")[: math.ceil(0.01 * K)]
        p.fill_(0.5 * density)
        p[rows] += 0.5 * density * K / len(rows)
    else:
        rows = torch.randperm(K, generator=gen, device="cuda")[: max(1, int(0.005 * K))]
        cols = torch.randperm(N, generator=gen, device="cuda")[: max(1, int(0.005 * N))]
        hot = len(rows) * N + len(cols) * K - len(rows) * len(cols)
        fill = min(0.75, 0.8 * density * K * N / hot)
        p.fill_((density * K * N - fill * hot) / (K * N - hot))
        p[rows] = fill
        p[:, cols] = fill
    hit = torch.rand(K, N, generator=gen, device="cuda") < p
    k, n = torch.nonzero(hit, as_tuple=True)
    return k, n


def _outlier_values(gen, count):
    """+-(6 to 20) standard deviations of the weights, in BF16."""
    v = synth.SIGMA * (6 + 14 * torch.rand(count, generator=gen, device="cuda"))
    return (v * (2 * torch.randint(0, 2, (count,), generator=gen, device="cuda") - 1)).to(torch.bfloat16)


def _codes(gen, L, k, n, zero):
    """Packed codes as quantised normal weights give them (bell-shaped around the zero-point, which is what an outlier's
    place holds), drawn on the GPU in the packed order: a nibble's place does not matter to an identically
    distributed code, and the outliers' places follow the word order that fq.h describes."""
    K, N, BN = L.K, L.N, L.BN
    q = (7.5 + 2.4 * torch.randn(K * N, generator=gen, device="cuda", dtype=torch.float16)).round_().clamp_(0, 15).to(torch.uint8)
    if k.numel():
        kr, c = k % 128, n % BN
        word = ((n // BN) * (K // 128) + k // 128) * 16 * BN + ((kr // 32) * BN + c) * 4 + (kr // 8) % 4
        q[word * 8 + (kr // 2) % 4 + 4 * (kr % 2)] = zero[k // L.group, n].to(torch.uint8)
    q = q.view(-1, 8)
    words = torch.zeros(q.shape[0], dtype=torch.int32, device="cuda")
    for i in range(8):
        words |= q[:, i].to(torch.int32) << (4 * i)
    return words


def _layer(gen, K, N, group, density, layout):
    """One packed layer on the GPU, as a model that was quantised before is loaded."""
    L = fq.fq_get_layout(K, N, group)
    k, n = _outlier_positions(gen, K, N, density, layout)
    v = _outlier_values(gen, k.numel())
    scale = (synth.SIGMA * (0.36 + 0.06 * torch.rand(K // group, N, generator=gen, device="cuda"))).to(torch.bfloat16)
    zero = torch.randint(6, 10, (K // group, N), generator=gen, device="cuda").to(torch.bfloat16)
    wq = _codes(gen, L, k, n, zero)
    indptr, info, packed = fq.fq_encode_tilecoo(L, k.to(torch.int32).cpu().numpy().view(np.uint32),
                                                n.to(torch.int32).cpu().numpy().view(np.uint32),
                                                v.view(torch.int16).cpu().numpy().view(np.uint16))
    if packed.shape[0] == 0:
        packed = np.zeros((8, 16), dtype=np.uint8)
    return dict(L=L, wq=wq, scale=scale, zero=zero, indptr=torch.from_numpy(indptr.view(np.int32)).cuda(),
                info=torch.from_numpy(info.view(np.int32)).cuda(), packed=torch.from_numpy(packed).cuda())


def _shapes(case):
    return BLOCK if case["kind"] == "block" else [(case["K"], case["N"])]


def prepare(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    if case["kind"] == "pack":
        K, N = case["K"], case["N"]
        W = synth.SIGMA * torch.randn(K, N, generator=gen, device="cuda")
        # The number of packets depends on the positions: they are the case's own, moved by whole tiles with the seed,
        # so that the packed arrays of two seeds can be compared.
        fixed = torch.Generator(device="cuda")
        fixed.manual_seed(K + N)
        k, n = _outlier_positions(fixed, K, N, case["density"], case["layout"])
        k, n = (k + 128 * (seed % (K // 128))) % K, (n + 256 * (seed // 7)) % N
        v = _outlier_values(gen, k.numel())
        W[k, n] = v.float()
        mask = torch.zeros(K, N, dtype=torch.uint8, device="cuda")
        mask[k, n] = 1
        return dict(case=case, W=W.cpu().numpy(), mask=mask.cpu().numpy(), k=k.to(torch.int32).cpu().numpy().view(np.uint32),
                    n=n.to(torch.int32).cpu().numpy().view(np.uint32), v=v.view(torch.int16).cpu().numpy().view(np.uint16))
    M = case["M"]
    calls = []
    for K, N in _shapes(case):
        c = _layer(gen, K, N, case["group"], case["density"], case["layout"])
        c["X"] = torch.randn(M, K, generator=gen, device="cuda").to(torch.bfloat16)
        c["Y"] = torch.empty(M, N, dtype=torch.bfloat16, device="cuda")
        if case["host"]:
            c["Xh"] = c["X"].cpu().pin_memory()
            c["Yh"] = torch.empty(M, N, dtype=torch.bfloat16).pin_memory()
        calls.append(c)
    ws = torch.zeros(max(fq.fq_workspace_bytes(c["L"], M) for c in calls), dtype=torch.uint8, device="cuda")
    return dict(case=case, M=M, calls=calls, ws=ws)


# --------------------------------------------------------------------------------------------------------- a pass

def run(state):
    case = state["case"]
    if case["kind"] == "pack":
        L = fq.fq_get_layout(case["K"], case["N"], case["group"])
        return [*fq.fq_pack_int4(L, state["W"], state["mask"]), *fq.fq_encode_tilecoo(L, state["k"], state["n"], state["v"])]
    M, ws = state["M"], state["ws"]
    if case["host"]:
        for c in state["calls"]:
            fq.fq_fused_host_io_async(c["L"], c["Xh"], M, c["X"], c["wq"], c["scale"], c["zero"], c["indptr"], c["info"],
                                      c["packed"], c["Y"], c["Yh"], ws)
        torch.cuda.current_stream().synchronize()      # the step's results are read on the host
        return [c["Yh"] for c in state["calls"]]
    for c in state["calls"]:
        fq.fq_fused_w4a16_outlier_gemm(c["L"], c["X"], M, c["wq"], c["scale"], c["zero"], c["indptr"], c["info"], c["packed"],
                                       c["Y"], ws)
    return [c["Y"] for c in state["calls"]]


def work(case):
    """Codes, scales and zero-points, the outliers by the paper's storage formula (descriptors, and four bytes for each
    outlier: no padding), X in and Y out.  For packing: the matrix and its mask in, the packed arrays out."""
    M, g, total = case["M"], case["group"], 0
    flops = 0
    for K, N in _shapes(case):
        bn = 256 if N % 256 == 0 else 128
        tiles = (K // 128) * (N // bn)
        stored = K * N // 2 + 4 * (K // g) * N + (tiles + 1) * 4 + tiles * (bn // 4) * 4 + 4 * round(case["density"] * K * N)
        if case["kind"] == "pack":
            total += stored + 5 * K * N + 10 * round(case["density"] * K * N)
            flops += 4 * K * N              # range (two comparisons), quotient, rounding
        else:
            total += stored + 2 * M * (K + N)
            flops += 2 * M * K * N
    return {"bytes": total, "flops": flops}


def tolerance(case):
    if case["kind"] == "pack":
        return "exact"
    # sums in FP32, one rounding to BF16: two correct results are at most one BF16 step apart (2^-8 of the value), and
    # somewhat more of a value that is small beside the others because its sum cancelled
    return {"rel": 4e-3, "max": 1.6e-2}
