"""No C++ exception leaves klmc_cluster_histogram: a program whose operator new throws gets
the same histogram (histogram_without_memory.cpp)."""
import os
import subprocess

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1309_4349_gb300 as klmc  # noqa: E402

HERE = os.path.dirname(os.path.abspath(__file__))


def test_histogram_without_host_memory(tmp_path):
    so = klmc.build()
    exe = str(tmp_path / "histogram_without_memory")
    subprocess.run(["g++", "-O1", "-std=c++17", "-I" + os.path.join(os.path.dirname(HERE), "include"),
                    os.path.join(HERE, "histogram_without_memory.cpp"), so, "-Wl,-rpath," + os.path.dirname(so), "-o", exe],
                   check=True)
    res = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    assert res.returncode == 0 and res.stdout == "same\n", (res.returncode, res.stderr)
