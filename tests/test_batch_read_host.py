"""The order of ts_batch_read's work and the calls of a load, over a fake of the CUDA runtime with two
devices (no GPU needed)."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CUDA = "/usr/local/cuda"


def test_reads_and_loads_over_a_fake_runtime(tmp_path):
    """The copies of a read are made on the batch's device, behind its pack
    kernel, whichever device is current; and a reader whose stream is busy
    holds up no other reader.  A load makes one allocation and one copy."""
    if not shutil.which("g++") or not os.path.exists(os.path.join(CUDA, "include", "cuda_runtime.h")):
        pytest.skip("needs g++ and the CUDA headers")
    from paper_2604_09221_gb300 import build
    lib = build.build()
    exe = tmp_path / "run"
    subprocess.run(["g++", "-std=c++17", "-O1", "-rdynamic", f"-I{os.path.join(ROOT, 'include')}",
                    f"-I{CUDA}/include", "-o", str(exe), os.path.join(HERE, "host", "run_batch_read.cpp"),
                    lib, f"-Wl,-rpath,{os.path.dirname(lib)}", f"-Wl,-rpath,{CUDA}/lib64",
                    f"-Wl,-rpath-link,{CUDA}/lib64", "-lpthread"], check=True, capture_output=True)
    out = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert out.returncode == 0, (out.returncode, out.stdout, out.stderr)
