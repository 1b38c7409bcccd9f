"""The build option of blocks of 8 phases for resident sweeps (-DKLMC_MAX_BLOCK=8 in
KLMC_NVCC_FLAGS): a library built with it gives the oracle's trajectories too."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1309_4349_gb300 as klmc  # noqa: E402
from paper_1309_4349_gb300 import _build  # noqa: E402

klmc.build()

RUN = """
import sys
import numpy as np
import oracle
import paper_1309_4349_gb300 as klmc
klmc.LIB_PATH = sys.argv[1]
for Lx, Ly, cluster, threads in ((100, 96, 4, 256), (257, 150, 8, 512), (70, 70, 2, 128)):
    for geometry in (klmc.TRI6, klmc.SQ4):
        lat = klmc.Lattice(Lx, Ly, geometry=geometry, n_A=Lx * Ly // 3, omega_over_kT=0.7, seed=5, cluster=cluster,
                           threads=threads)
        assert lat.plan() == 8
        lat.sweep(1)
        lat.sweep(4)
        ref = oracle.run(Lx, Ly, geometry, 0.7, 5, oracle.init(Lx, Ly, Lx * Ly // 3, 5), 0, 5)
        assert np.array_equal(lat.get_lattice(), ref.lattice)
        assert lat.energy()[0] == ref.n_unlike
        lat.close()
"""


def test_blocks_of_eight_phases(tmp_path):
    flags = _build.ARCH + ["-O3", "-std=c++17", "-Xcompiler", "-fPIC"]
    obj, so = str(tmp_path / "sweep_resident.o"), str(tmp_path / "libklmc8.so")
    subprocess.run([_build._nvcc()] + flags + ["-DKLMC_MAX_BLOCK=8", "-I" + os.path.join(_build.ROOT, "include"),
                                               "-I" + _build.CSRC, "-c", os.path.join(_build.CSRC, "sweep_resident.cu"),
                                               "-o", obj], check=True)
    rest = [os.path.join(_build.OBJ, s.replace(".cu", ".o")) for s in _build.SOURCES if s != "sweep_resident.cu"]
    subprocess.run([_build._nvcc()] + _build.ARCH + ["-shared", "-o", so, obj] + rest, check=True)
    res = subprocess.run([sys.executable, "-c", RUN, so], cwd=_build.ROOT, capture_output=True, text=True, timeout=300)
    assert res.returncode == 0, res.stderr
