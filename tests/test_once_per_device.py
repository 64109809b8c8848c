"""Settings of a kernel that belong to one device (the dynamic shared-memory limit)
are made on every device the process uses, not once per process."""
import glob
import os
import re
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_1211_1645_gb300", "csrc")


def test_once_per_device_host(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    out = str(tmp_path / "once_host")
    subprocess.check_call([nvcc, "-O2", "-std=c++17", "-Xcompiler", "-pthread", "-I" + CSRC, "-o", out,
                           os.path.join(HERE, "host", "once_per_device_host.cu")])
    assert subprocess.check_output([out], timeout=60).strip() == b"ok"


def test_no_device_attribute_is_set_once_per_process():
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh"))):
        text = open(path).read()
        assert "call_once" not in text, os.path.basename(path)
        # and its result is looked at
        assert not re.search(r"^\s*cudaFuncSetAttribute\(", text, re.M), os.path.basename(path)
