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
    build.build_pycall()
    assert not calls
    monkeypatch.setattr(torch, "__version__", "0.0.1")
    build.build_pycall()
    assert len(calls) == 1
    monkeypatch.setattr(fq, "_call", None)
    with pytest.raises(ImportError, match="built for"):
        fq._pycall()
