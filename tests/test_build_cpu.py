"""The build: what it leaves behind."""
import os
import shutil
import subprocess
import sys
import sysconfig

import pytest

import paper_2609_27085_b200 as cf
from paper_2609_27085_b200 import build as cf_build

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


def test_the_allocation_free_call_keeps_to_its_stack(tmp_path):
    """cf_decode_attention_static promises about 124 KB of stack: its own frame, and no other of its file worth mentioning (a plan
    that the launches carry is not copied on the way).  Frame sizes as the host compiler reports them."""
    src = os.path.join(ROOT, PKG, "csrc", "decode_splitk.cu")
    nvcc = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "bin", "nvcc")
    subprocess.run([nvcc if os.path.exists(nvcc) else "nvcc", "-gencode", "arch=compute_100a,code=compute_100a", "-Xcicc", "-O0", "-O3", "-std=c++17",
                    "-Xcompiler", "-fPIC,-fstack-usage", "--expt-relaxed-constexpr", "-c", src, "-o", str(tmp_path / "d.o")],
                   check=True, capture_output=True, timeout=600)
    frames = {}
    for line in (tmp_path / "d.su").read_text().splitlines():
        name, size, _ = line.split("\t")
        frames[name] = int(size)
    sizes = sorted(frames.values())                                   # the entry point's frame is the largest by far
    assert 112 * 1024 < sizes[-1] <= 126 * 1024 and sizes[-2] <= 4096, sizes[-3:]


def test_the_marshalling_extension_is_the_interpreters_own(monkeypatch):
    """Its name carries the ABI tag; an interpreter that it was not built for finds no file and says so."""
    assert cf_build.MARSHAL == cf.MARSHAL_PATH and cf.MARSHAL_PATH.endswith(sysconfig.get_config_var("EXT_SUFFIX"))
    cf_build.build()
    assert os.path.exists(cf.MARSHAL_PATH)
    monkeypatch.setattr(cf, "_lib", None)
    monkeypatch.setattr(cf, "MARSHAL_PATH", cf.MARSHAL_PATH.replace("cpython-", "cpython-9"))
    with pytest.raises(ImportError, match="is missing"):
        cf.load_library()
