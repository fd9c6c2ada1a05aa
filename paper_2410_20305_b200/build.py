"""Builds libpsa.so in-tree with nvcc for sm_100a (cross-compiles without a GPU)."""
from __future__ import annotations

import os
import subprocess
import sys

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libpsa.so")
LIB_DEBUG = os.path.join(HERE, "libpsa_debug.so")   # the same sources with -DPSA_DEBUG_BOUNDS (checked global indices)
SOURCES = ["psa_plan.cpp", "psa_host_helpers.cpp", "psa_api.cu", "psa_fwd.cu", "psa_bwd.cu", "psa_bwd_static.cu", "psa_selftest.cu",
           "dpo_logp.cu", "dpo_loss.cu", "psa_rope.cu"]


def _stale(lib=LIB) -> bool:
    if not os.path.exists(lib):
        return True
    t = os.path.getmtime(lib)
    deps = [os.path.join(CSRC, f) for f in os.listdir(CSRC) if f != "psa_native.cpp"] + [os.path.join(ROOT, "include", "psa.h")]
    return any(os.path.getmtime(d) > t for d in deps)


def build(force: bool = False, verbose: bool = False, debug: bool = False) -> str:
    """Builds libpsa.so, or with debug=True libpsa_debug.so: the same code with every index that a thread
    forms itself checked against its tensor (an out-of-range one sets PSA_DEVSTAT_OUT_OF_BOUNDS and is skipped)."""
    lib = LIB_DEBUG if debug else LIB
    if not force and not _stale(lib):
        return lib
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    cmd = [nvcc, "-O3", "-std=c++17", "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo",
           "-Xcompiler", "-fPIC", "-shared", "-I", os.path.join(ROOT, "include"), "-I", CSRC,
           "-o", lib] + [os.path.join(CSRC, s) for s in SOURCES]
    if debug:
        cmd += ["-DPSA_DEBUG_BOUNDS"]
    if verbose:
        cmd += ["-Xptxas", "-v"]
    res = subprocess.run(cmd, capture_output=True, text=True)
    if verbose or res.returncode != 0:
        sys.stderr.write(res.stdout + res.stderr)
    if res.returncode != 0:
        raise RuntimeError("nvcc failed building " + os.path.basename(lib))
    return lib


def native_path() -> str:
    """Where psa_native's library for this interpreter and this torch lies.  It has torch's tensor layout and CPython's
    ABI compiled in, so one that was built for others must never be loaded: they are part of its name."""
    import sysconfig
    import torch
    torch_tag = "".join(c if c.isalnum() or c in ".+" else "_" for c in torch.__version__)
    return os.path.join(HERE, "psa_native.torch-%s-abi%d%s" % (torch_tag, torch._C._GLIBCXX_USE_CXX11_ABI,
                                                             sysconfig.get_config_var("EXT_SUFFIX")))


def build_native(force: bool = False) -> str:
    """Builds the compiled route of the binding's calls (csrc/psa_native.cpp) against the torch that runs."""
    source, native = os.path.join(CSRC, "psa_native.cpp"), native_path()
    deps = [source, os.path.join(ROOT, "include", "psa.h")]

    def current():
        return os.path.exists(native) and all(os.path.getmtime(d) <= os.path.getmtime(native) for d in deps)

    if not force and current():
        return native
    import fcntl
    import sysconfig
    import torch
    with open(source) as lock:   # one process of a node builds, the others wait for it
        fcntl.flock(lock, fcntl.LOCK_EX)
        if not force and current():
            return native
        home = os.path.dirname(torch.__file__)
        cuda = os.path.dirname(os.path.dirname(os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")))
        include = [os.path.join(ROOT, "include"), os.path.join(home, "include"),
                   os.path.join(home, "include", "torch", "csrc", "api", "include"), sysconfig.get_paths()["include"],
                   os.path.join(cuda, "include")]
        # into place at once: another process may be about to load it
        out = "%s.%d.tmp" % (native, os.getpid())
        cmd = ["g++", "-O2", "-std=c++17", "-fPIC", "-shared", "-D_GLIBCXX_USE_CXX11_ABI=%d" % torch._C._GLIBCXX_USE_CXX11_ABI]
        cmd += [a for d in include for a in ("-I", d)] + ["-o", out, source, "-L", os.path.join(home, "lib")]
        cmd += ["-lc10", "-lc10_cuda", "-ltorch_cpu", "-ltorch_python"]
        res = subprocess.run(cmd, capture_output=True, text=True)
        if res.returncode != 0:
            raise RuntimeError("g++ failed building psa_native: " + res.stderr[-2000:])
        os.replace(out, native)
    return native


if __name__ == "__main__":
    print(build(force=True, verbose=True))
    print(build(force=True, debug=True))
    print(build_native(force=True))
