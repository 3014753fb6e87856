"""Runs a snippet against libspdba.so on the fake CUDA runtime of fake_cudart.c, in a process of
its own (no GPU, no torch)."""
import os
import shutil
import subprocess
import sys

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)

PRELUDE = """
import ctypes, sys
sys.path.insert(0, %r)
import numpy as np
from paper_2609_03922_gb300 import spdba
L = spdba.lib()
fake = ctypes.CDLL(%r)
for f in ("fake_foreign_launches", "fake_foreign_copies", "fake_launches", "fake_instantiated"):
    getattr(fake, f).restype = ctypes.c_long
"""


def run(tmp_path, snippet):
    from paper_2609_03922_gb300 import build
    cc = shutil.which("gcc") or shutil.which("cc")
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    inc = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")
    if cc is None or not os.path.exists(os.path.join(inc, "cuda_runtime_api.h")):
        pytest.skip("no C compiler or CUDA headers")
    build.build()
    so = str(tmp_path / "fake_cudart.so")
    subprocess.run([cc, "-std=c11", "-shared", "-fPIC", "-I", inc, os.path.join(HERE, "fake_cudart.c"), "-o", so],
                   check=True)
    r = subprocess.run([sys.executable, "-c", PRELUDE % (ROOT, so) + snippet], capture_output=True, text=True,
                       env=dict(os.environ, LD_PRELOAD=so), timeout=300)
    assert r.returncode == 0, r.stdout + r.stderr
    return r.stdout
