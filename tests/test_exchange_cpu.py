"""The halo exchange of the resident sweeps, its own code run on the host over a model of
the cluster (exchange_model.cpp): threads and stores held back by an adversary never
mix two blocks' rows and never leave a CTA waiting."""
import os
import subprocess

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_1309_4349_gb300", "csrc")


def test_exchange_against_adversaries(tmp_path):
    exe = str(tmp_path / "exchange_model")
    subprocess.run(["g++", "-O1", "-std=c++17", "-I" + CSRC, os.path.join(HERE, "exchange_model.cpp"), "-o", exe],
                   check=True)
    res = subprocess.run([exe], capture_output=True, text=True, timeout=300)
    assert res.returncode == 0, res.stdout
