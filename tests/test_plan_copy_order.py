"""Copies that the split schedule moves ahead of their GEMM, against the schedule builder itself."""
import os
import subprocess

from tests.conftest import ROOT
from tests.libtools import lib


def test_copies_ahead_of_their_gemm_meet_nothing_it_uses(tmp_path):
    lib()
    from paper_1005_0088_gb300 import build as b
    exe = str(tmp_path / "order")
    objs = [os.path.join(b.BUILD, o) for o in ("split_gemm.cu.o", "analyze.cpp.o", "plan_check.cpp.o", "mu_search.cpp.o")]
    cmd = [b._nvcc()] + b.ARCH + ["-std=c++17", "-O1", "-I" + b.INCLUDE, "-I" + b.CSRC,
                                  os.path.join(ROOT, "tests", "plan_copy_order.cpp")] + objs + ["-lpthread", "-o", exe]
    res = subprocess.run(cmd, capture_output=True, text=True)
    assert res.returncode == 0, res.stderr
    out = subprocess.run([exe], capture_output=True, text=True)
    print(out.stdout)
    assert out.returncode == 0, out.stdout
