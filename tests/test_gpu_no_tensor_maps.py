"""A float64 context whose tensor maps cannot be encoded is built all the same and runs on the CUDA cores: the encoder is
replaced by one that refuses, in a process of its own (the library's own symbol, preloaded)."""
import os
import subprocess
import sys

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

REFUSE = "int _ZN3fmi8encode3tEP14CUtensorMap_stPKv24CUtensorMapDataType_enumiiiiii(void) { return 0; }\n"
RUN = """
import torch
import paper_2005_05398_gb300 as pkg
from fm_inputs import make_workload, rand_vec
out = []
for mma in (0, 1):
    ctx = pkg.Context(make_workload("He", 1, nint=(9, 7, 3), R=(20.0, 17.0)), mma=mma, restart_m=4, ncv=4)
    ctx.fm_set_shift(-2.4)
    v = torch.tensor(rand_vec(ctx.n, 2), device="cuda")
    y = torch.empty_like(v)
    ctx.fm_precond_apply(v, y)
    torch.cuda.synchronize()
    out.append(y)
assert torch.equal(out[0], out[1])
print("same kernels")
"""


def test_float64_context_without_tensor_maps(tmp_path):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    src, so = tmp_path / "refuse.c", tmp_path / "refuse.so"
    src.write_text(REFUSE)
    subprocess.run(["gcc", "-shared", "-fPIC", "-o", str(so), str(src)], check=True)
    r = subprocess.run([sys.executable, "-c", RUN], cwd=ROOT, env=dict(os.environ, LD_PRELOAD=str(so), PYTHONPATH=ROOT),
                       capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and "same kernels" in r.stdout, r.stderr[-1500:]
