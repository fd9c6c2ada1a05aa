"""What programmatic dependent launch asks of the kernels and of their launches, checked without a GPU."""
import os
import re
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2410_20305_b200", "csrc")

CALL = r"""
#include "psa_launch.cuh"
__global__ void kernel(const float* x, int* n, long long rows) {}
void f(const float* x, float* y, int* n, cudaStream_t s) { psa::launch_behind(true, kernel, dim3(1), 32, 0, s, %s); }
"""


@pytest.mark.parametrize("arguments,fits", [("x, n, 5", True), ("y, n, 5LL", True), ("x, y, 5", False), ("n, n, 5", False), ("5LL, n, 5", False)])
def test_arguments_convert_as_in_a_launch(tmp_path, arguments, fits):
    """Only conversions that <<<>>> makes too: a pointer of another type, or a number for one, does not compile."""
    (tmp_path / "call.cu").write_text(CALL % arguments)
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    run = subprocess.run([nvcc, "-std=c++17", "-gencode", "arch=compute_100a,code=sm_100a", "-I", CSRC, "-c", str(tmp_path / "call.cu"),
                          "-o", str(tmp_path / "call.o")], capture_output=True, text=True)
    assert (run.returncode == 0) == fits, run.stderr


def test_what_the_kernel_before_may_write_is_not_promised_to_be_read_only():
    """`const T* __restrict__` says that nobody writes there while the kernel runs, and lets the compiler load ahead of
    behind_wait(), or through the path that is not coherent.  A kernel that starts while its producer still runs must not
    say so.  (dpo_logp_kernel starts behind the kernel that clears its sums, which has waited for the logits.)"""
    seen = []
    for name in sorted(os.listdir(CSRC)):
        if not name.endswith(".cu"):
            continue
        for part in re.split(r"(?=__global__)", open(os.path.join(CSRC, name)).read())[1:]:
            head, body = part.split("{", 1)
            kernel = re.search(r"(\w+_kernel)\s*\(", head)
            end = re.search(r"^}", body, re.M)
            if not kernel or "behind_wait();" not in body[:end.start()]:
                continue
            seen.append(kernel.group(1))
            if kernel.group(1) != "dpo_logp_kernel":
                assert not re.search(r"const [^,*]*\* __restrict__", head), kernel.group(1)
    assert set(seen) >= {"psa_fwd_kernel", "psa_bwd_kernel", "psa_bwd_delta_kernel", "psa_bwd_convert_kernel", "dpo_logp_kernel",
                         "dpo_logp_bwd_kernel", "dpo_loss_kernel", "simpo_loss_kernel", "orpo_loss_kernel"}
