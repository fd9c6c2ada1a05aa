"""The compiled route of the binding (psa_native.cpp) where there is no GPU: how it is built and loaded, and that it leaves
every call that it does not take to binding.py."""
import os
import subprocess
import sys

import pytest

from paper_2410_20305_b200 import build

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
B._load_native()
a = lambda *x: np.array(x, dtype=np.int32)
print(B._native.plan(a(0, 10), a(4), a(3), a(3), 4, 2, 64, 0.0))
""").split() == ["None"]


@pytest.mark.parametrize("other", [("torch.__version__", "99.1.0+cu1"), ("torch._C._GLIBCXX_USE_CXX11_ABI", 7)])
def test_a_library_of_another_torch_or_interpreter_is_not_taken(monkeypatch, other):
    import sysconfig
    here = build.build_native()
    assert os.path.exists(here) and build.build_native() == here
    monkeypatch.setattr(other[0], other[1])
    elsewhere = build.native_path()
    assert elsewhere != here and not os.path.exists(elsewhere)
    monkeypatch.undo()
    suffix = sysconfig.get_config_var("EXT_SUFFIX")
    assert here.endswith(suffix)   # the interpreter's ABI and platform
    monkeypatch.setattr(sysconfig, "get_config_var", lambda name: ".cpython-399" + suffix if name == "EXT_SUFFIX" else None)
    assert build.native_path() not in (here, elsewhere)


def test_calls_on_the_host_alone_need_neither_torch_nor_a_compiler():
    assert _python("""
import sys, subprocess
from paper_2410_20305_b200 import binding as B
B.load_library()
subprocess.run = None      # nothing is built from here on
B.psa_pack_ffd([5, 7, 3], 10)
B.psa_pack_ffd_emit([5, 7], [1, 1], [1, 1], 20)
B.psa_logp_labels(range(9), [0, 9], [3], [3], [3])
B.psa_position_ids([0, 9], [3], [3], [3])
B.psa_plan([0, 9], [3], [3], [3], 4, 2, 64, host_only=True).close()
print("torch" in sys.modules, B._native, B._native_tried)
""").split() == ["False", "None", "False"]


def test_a_route_that_cannot_be_had_is_said_once_and_the_calls_go_on():
    assert _python("""
import warnings
from paper_2410_20305_b200 import binding as B, build
def fails():
    raise RuntimeError("no compiler here")
build.build_native = fails
B._cuda_ready = lambda: True
with warnings.catch_warnings(record=True) as said:
    warnings.simplefilter("always")
    for _ in range(3):
        B.psa_pack_ffd([5, 7, 3], 10)
print(len(said), "no compiler here" in str(said[0].message), said[0].category.__name__, B._native)
""").split() == ["1", "True", "RuntimeWarning", "None"]
