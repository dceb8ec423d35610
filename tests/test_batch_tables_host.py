"""The batch's tile tables against a fake of the CUDA runtime (tests/native/batch_tables_host.cpp): what a
launch was given stays as it is until the batch is destroyed, and running out of memory is an error that
leaves the batch as it was."""
import os
import shutil
import subprocess

import pytest

from paper_1703_04594_gb300 import lbm
from tests.gpu_util import ensure_built

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    ensure_built()
    nvcc = os.path.realpath(shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc")
    include = os.path.join(os.path.dirname(os.path.dirname(nvcc)), "include")
    exe = str(tmp_path_factory.mktemp("batch") / "batch_tables_host")
    libdir, lib = os.path.split(lbm.LIB_PATH)
    subprocess.run(["g++", "-std=c++17", "-rdynamic", "-I", include, "-o", exe,
                    os.path.join(HERE, "native", "batch_tables_host.cpp"), "-L", libdir, "-l:" + lib,
                    "-Wl,-rpath," + libdir, "-Wl,--allow-shlib-undefined"], check=True, capture_output=True)
    return exe


@pytest.mark.parametrize("what", ["in_flight", "no_device_memory", "no_host_memory", "plan"])
def test_tables(program, what):
    out = subprocess.run([program, what], capture_output=True, text=True, timeout=60)
    assert (out.returncode, out.stdout.strip()) == (0, "ok"), out.stderr
