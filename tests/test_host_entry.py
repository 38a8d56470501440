"""The entries from the host: what they do with arguments that are no good, and with values at the edge of a type.  CPU only."""
import os
import subprocess
import sys

import pytest

from paper_2608_15531_b200 import binding as fq

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

_BATCHED_TENSOR = """
import torch
from torch._subclasses.fake_tensor import FakeTensorMode
from paper_2608_15531_b200 import binding as fq
L = fq.fq_get_layout(128, 128, 128)
with FakeTensorMode():
    t = torch.empty(2, 128, dtype=torch.int16, device="cuda")
for call in (lambda x: fq.fq_fused_w4a16_outlier_gemm(L, x, 1, t, t, t, t, t, t, t, t),
             lambda x: fq.fq_fused_host_io_async(L, torch.empty(1), 1, x, t, t, t, t, t, t, t, torch.empty(1), t)):
    try:
        torch.func.vmap(lambda x: (call(x), x)[1])(t)
    except RuntimeError as e:
        print("refused:", "storage" in str(e))
"""


def test_a_tensor_without_storage_is_a_python_error():
    """What the tensor library throws must not leave the CPython entry (the process would end)."""
    p = subprocess.run([sys.executable, "-c", _BATCHED_TENSOR], cwd=ROOT, capture_output=True, text=True)
    assert p.returncode == 0 and p.stdout.split("\n")[:2] == ["refused: True"] * 2, (p.returncode, p.stdout, p.stderr[-500:])


@pytest.mark.parametrize("field,value", [("abi", 7), ("BK", 0), ("BK", 1), ("BN", 0), ("buckets_per_tile", 2 ** 31), ("K", 0)])
def test_the_encoder_refuses_a_bad_layout_before_it_makes_arrays(field, value):
    L = fq.fq_get_layout(1 << 20, 1 << 18, 128)
    setattr(L, field, value)
    with pytest.raises(fq.FqError) as e:
        fq.fq_encode_tilecoo(L, [], [], [])
    assert e.value.code == fq.FQ_ERR_INVALID_ARG


def test_the_entry_belongs_to_the_torch_it_was_built_for(monkeypatch):
    """Another torch version: the binding refuses the old build, and the build step sees that it is stale."""
    import torch
    from paper_2608_15531_b200 import build
    assert fq._pycall().built_for == f"torch {torch.__version__}"
    calls = []
    monkeypatch.setattr(build.subprocess, "run", lambda cmd, **kw: calls.append(cmd))
    monkeypatch.setattr(build, "stale", lambda *a: False)      # (whatever the sources' times)
    build.build_pycall()
    assert not calls
    monkeypatch.setattr(torch, "__version__", "0.0.1")
    build.build_pycall()
    assert len(calls) == 1
    monkeypatch.setattr(fq, "_call", None)
    with pytest.raises(ImportError, match="built for"):
        fq._pycall()


_PACK = """
import sys, numpy as np
from paper_2608_15531_b200 import binding as fq
fq.LIB_PATH = sys.argv[1]
fq.EXPORTS = [n for n in fq.EXPORTS if n in ("fq_get_layout", "fq_pack_int4", "fq_pack_int4_sizes", "fq_last_error")]
K, N = 128, 256
W = (0.02 * np.random.default_rng(0).standard_normal((K, N))).astype(np.float32)
mask = np.zeros((K, N), dtype=np.uint8)
W[:, 0] = 0.0                                       # degenerate: 0 / 0
W[:, 1] *= 1e-38; W[5, 1] = 3e38; mask[5, 1] = 1    # an outlier over a tiny scale: beyond any integer
W[:, 2] = 0.0; W[9, 2] = 7.0; mask[9, 2] = 1        # nothing but an outlier: 7 / 0
W[3, 3] = np.inf; W[4, 4] = -np.inf; W[6, 5] = np.nan
out = fq.fq_pack_int4(fq.fq_get_layout(K, N, 128), W, mask)
sys.stdout.write("".join(a.tobytes().hex() for a in out))
"""


def test_packing_converts_only_what_an_integer_holds(tmp_path):
    """The packer under -fsanitize=float-cast-overflow: quotients that are no numbers, infinite, or too large for an integer are settled
    before they are converted.  The arrays are those of the library."""
    lib = str(tmp_path / "libfq_ubsan.so")
    subprocess.run(["g++", "-O1", "-std=c++17", "-fPIC", "-shared", "-fopenmp", "-ffp-contract=off", "-fsanitize=float-cast-overflow",
                    "-fno-sanitize-recover=all", "-I", os.path.join(ROOT, "include"), os.path.join(ROOT, "paper_2608_15531_b200", "csrc", "fq_host.cpp"),
                    "-o", lib], check=True)
    runs = [subprocess.run([sys.executable, "-c", _PACK, path], cwd=ROOT, capture_output=True, text=True) for path in (lib, fq.LIB_PATH)]
    assert runs[0].returncode == 0, runs[0].stderr
    assert runs[1].returncode == 0 and runs[0].stdout and runs[0].stdout == runs[1].stdout
