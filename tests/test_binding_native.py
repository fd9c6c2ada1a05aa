"""The compiled route of the binding (psa_native.cpp) where there is no GPU: how it is built and loaded, and that it leaves
every call that it does not take to binding.py."""
import os
import subprocess
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _python(code, **env):
    """What a fresh interpreter without a GPU prints."""
    run = subprocess.run([sys.executable, "-c", code], cwd=ROOT, capture_output=True, text=True, timeout=600,
                         env={**os.environ, "CUDA_VISIBLE_DEVICES": "", **env})
    assert run.returncode == 0, run.stderr[-2000:]
    return run.stdout


def test_plan_without_a_device_is_left_to_the_binding():
    # the current stream cannot be had: a C++ exception, which must not leave the extension
    assert _python("""
import numpy as np
from paper_2410_20305_b200 import binding as B
B.load_library()
a = lambda *x: np.array(x, dtype=np.int32)
print(B._native.plan(a(0, 10), a(4), a(3), a(3), 4, 2, 64, 0.0))
""").split() == ["None"]
