"""What the library asks of the CUDA runtime, without a GPU: a preloaded fake
runtime (fake_cudart.cpp) writes the calls down instead of running kernels."""
import os
import re
import subprocess
import sys

import pytest

from paper_1910_04358_gb300 import build

HERE = os.path.dirname(os.path.abspath(__file__))
CUDA = os.path.dirname(os.path.dirname(build._nvcc()))

PRELUDE = """
import ctypes, sys
import numpy as np
from paper_1910_04358_gb300 import rambo
log = ctypes.CDLL(None).fake_cudart_log
log.restype = ctypes.c_char_p
ptr = lambda a: a.ctypes.data
def aligned(nbytes):
    a = np.zeros(nbytes + 256, np.uint8)
    return a[-ptr(a) % 256:][:nbytes]
"""


@pytest.fixture(scope="module")
def calls(tmp_path_factory):
    """calls(code): the lines that the fake runtime wrote while `code` ran."""
    so = str(tmp_path_factory.mktemp("fake") / "fake_cudart.so")
    subprocess.run(["g++", "-std=c++17", "-shared", "-fPIC", f"-I{CUDA}/include", os.path.join(HERE, "fake_cudart.cpp"),
                    "-o", so], check=True)
    build.build()

    def run(code):
        r = subprocess.run([sys.executable, "-c", PRELUDE + code], cwd=os.path.dirname(HERE), text=True,
                           capture_output=True, env=dict(os.environ, LD_PRELOAD=so))
        assert r.returncode == 0, r.stderr
        return r.stdout.splitlines()
    return run


def _stream(line):
    return re.search(r"stream=(\S+)", line).group(1)


def test_set_partition_makes_the_patterns_behind_the_copy(calls):
    lines = calls("""
idx = rambo.Index(100, 32, 4, 256, 2)
log()
idx.set_partition(np.zeros((100, 4), np.uint32))
print(log().decode())
""")
    copy, launch = [l for l in lines if l]
    assert copy.startswith("copy bytes=1600") and "k_patterns" in launch
    assert "stream=" in copy and _stream(copy) == _stream(launch)
