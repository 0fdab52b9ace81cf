"""What the C ABI cannot reach of the device code, through a small library
compiled from it: waits that run out, tables that are full."""

import ctypes
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))


def _compile(tmp, name, *defines):
    from paper_2411_11244_gb300 import build as B
    out = os.path.join(tmp, name + ".so")
    src = [os.path.join(HERE, "native", "device_checks.cu"), os.path.join(B.CSRC, "gd_build.cu")]
    cmd = [B.nvcc(), *B.FLAGS, *B.ARCH, *defines, "-I", B.CSRC, "-shared", "-o", out, *src]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return ctypes.CDLL(out)


@pytest.fixture(scope="module")
def checks(tmp_path_factory):
    return _compile(str(tmp_path_factory.mktemp("native")), "checks")


@pytest.mark.parametrize("n", [1025, 100_003, 300_001])
def test_sort_that_gives_up_writes_nothing(checks, n):
    """A tile of the first pass never publishes: the waits for it run out, the
    passes that follow leave their buffers alone (the pairs that the first pass
    did not write would be placed beyond them), and the error word is set."""
    rng = np.random.default_rng(n)
    keys = rng.integers(0, 1 << 63, n, dtype=np.uint64)
    p = keys.ctypes.data_as(ctypes.c_void_p)
    assert checks.check_sort_gives_up(p, ctypes.c_longlong(n), 4) == 0
