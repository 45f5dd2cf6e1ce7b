"""The upload of a master's POLC matrix, on a stand-in for the CUDA runtime (CPU only, see
fake_cuda/master_upload.cpp): the host copy of P lives until the asynchronous copy from it
has ended."""
import os
import shutil
import subprocess

import pytest

from paper_1903_01852_gb300 import build

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
WRAPPED = ["GetDeviceCount", "SetDevice", "GetLastError", "StreamCreateWithPriority", "StreamDestroy", "StreamSynchronize",
           "EventCreateWithFlags", "EventDestroy", "Malloc", "Free", "HostAlloc", "FreeHost", "Memset", "Memcpy", "MemcpyAsync"]


def test_host_memory_outlives_the_copies_from_it(tmp_path):
    if not (shutil.which("nvcc") or os.path.exists("/usr/local/cuda/bin/nvcc")):
        pytest.skip("nvcc not available")
    objs = []
    for src in (os.path.join(build.CSRC, "rtc_master.cu"), os.path.join(ROOT, "tests", "fake_cuda", "master_upload.cpp")):
        objs.append(str(tmp_path / (os.path.basename(src) + ".o")))
        subprocess.run([build.nvcc(), "-std=c++17", "-O1", *build.ARCH, "-I", os.path.join(ROOT, "include"),
                        "-I", build.CSRC, "-c", src, "-o", objs[-1]], check=True)
    exe = str(tmp_path / "master_upload")
    wraps = [a for n in WRAPPED for a in ("-Xlinker", "--wrap=cuda" + n)]
    subprocess.run([build.nvcc(), *build.ARCH, *objs, *wraps, "-o", exe], check=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout + r.stderr
