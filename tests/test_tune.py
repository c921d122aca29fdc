"""The autotuner's choice between the two GEMM paths, against planted times."""
import os
import shutil
import subprocess

import pytest

from tests.conftest import ROOT


def test_paths_are_chosen_with_the_steps_they_depend_on(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no C++ compiler")
    csrc = os.path.join(ROOT, "paper_1005_0088_gb300", "csrc")
    exe = str(tmp_path / "tune")
    subprocess.run([gxx, "-std=c++17", "-O1", "-I" + csrc, os.path.join(ROOT, "tests", "tune_check.cpp"),
                    os.path.join(csrc, "tune.cpp"), "-o", exe], check=True, capture_output=True, text=True)
    out = subprocess.run([exe], capture_output=True, text=True)
    print(out.stdout)
    assert out.returncode == 0, out.stdout
