"""What the launch wrapper of the kernels (sa_launch) takes and refuses at compile time.  Needs nvcc, no GPU."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SOURCE = """
#include "sa_device.cuh"
__global__ void kernel(const int32_t *index, int32_t *status, float *out, int64_t n)
{
    sa_after_previous();
    if (n > 0) out[0] = float(index[0] + status[0]);
}
__global__ void copy(%s in, float *out)
{
    const sa_ready ready = sa_after_previous();
    (void)ready;
    out[0] = %s;
}
cudaError_t launch(const int32_t *index, int32_t *status, float *out, const float *in)
{
    cudaError_t e = sa_launch(copy, 1u, 32u, 0, nullptr, in, out);
    if (e != cudaSuccess) return e;
    return sa_launch(kernel, 1u, 32u, 0, nullptr, %s);
}
"""


def _compiles(tmp_path, args="index, status, out, int64_t(7)", in_type="sa_input", read="ready(in).ld()"):
    src = tmp_path / "launch.cu"
    src.write_text(SOURCE % (in_type, read, args))
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    r = subprocess.run([nvcc, "-gencode", "arch=compute_100a,code=sm_100a", "-std=c++17", "-I", os.path.join(ROOT, "include"),
                        "-I", os.path.join(ROOT, "paper_2311_09549_b200", "csrc"), "-c", str(src), "-o", str(tmp_path / "launch.o")],
                       capture_output=True, text=True, timeout=300)
    return r.returncode == 0, r.stderr


@pytest.mark.parametrize("args, right", [
    ("index, status, out, 7", True),                  # int -> int64_t, as in a call
    ("index, out, status, int64_t(7)", False),        # two arguments swapped
    ("index, index, out, int64_t(7)", False),         # a constant array where the kernel writes
    ("index, status, int64_t(7), out", False),        # a number for a pointer
])
def test_arguments_convert_only_as_in_a_call(tmp_path, args, right):
    ok, log = _compiles(tmp_path, args)
    assert ok == right, log


@pytest.mark.parametrize("in_type, read, right", [
    ("sa_input", "ready(in).ld()", True),
    ("sa_values", "in.p[0]", True),
    ("const float *", "in[0]", False),                # would be read as data that nothing writes while the kernel lives
    ("const float *__restrict__", "__ldg(in)", False),
])
def test_numbers_that_a_kernel_may_have_written_are_not_read_as_constants(tmp_path, in_type, read, right):
    """A kernel that starts beside the one before it may not read that one's results through the read-only path."""
    ok, log = _compiles(tmp_path, in_type=in_type, read=read)
    assert ok == right, log
    if not right:
        assert "fp32 inputs are sa_input or sa_values" in log


@pytest.mark.parametrize("read", ["in.ld()", "sa_data(in.p, 0).ld()"])
def test_such_numbers_cannot_be_loaded_without_having_waited(tmp_path, read):
    assert not _compiles(tmp_path, read=read)[0]
