"""The build: what it leaves behind."""
import os
import shutil
import subprocess
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
PKG = "paper_2609_27085_b200"


def test_a_failed_build_leaves_no_temporaries(tmp_path):
    """nvcc fails (a stand-in that exits with 1) while g++ succeeds: nothing but the sources and the object folder is left."""
    shutil.copytree(os.path.join(ROOT, PKG, "csrc"), tmp_path / PKG / "csrc")
    shutil.copytree(os.path.join(ROOT, "include"), tmp_path / "include")
    shutil.copy(os.path.join(ROOT, PKG, "build.py"), tmp_path / PKG)
    before = set(os.listdir(tmp_path / PKG)) | {"build", "__pycache__"}
    nvcc = tmp_path / "cuda" / "bin" / "nvcc"
    nvcc.parent.mkdir(parents=True)
    nvcc.write_text("#!/bin/sh\nexit 1\n")
    nvcc.chmod(0o755)
    r = subprocess.run([sys.executable, str(tmp_path / PKG / "build.py"), "--force"], env=dict(os.environ, CUDA_HOME=str(tmp_path / "cuda")),
                       capture_output=True, text=True, timeout=300)
    assert r.returncode != 0
    assert set(os.listdir(tmp_path / PKG)) <= before
