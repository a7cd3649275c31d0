"""Rules by which the host chooses between two forms of a kernel, at limits that no trace of a test reaches: a program of its own
includes the library's header and compares each rule with the arithmetic that the kernel does."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include "il_internal.h"
#include <stdio.h>
int main()
{
    // Two streams of one row: the second one's tail is a 32-bit count of bytes from the first one's start (as in the kernel).
    const int64_t most = INT64_C(1) << 29;
    const int64_t at[] = {0, 2, 1000, most / 2, most - 4, most - 2, most - 1, most, most + 2, 2 * most, 3 * most + 6};
    for (int64_t off_a : at) for (int64_t d : at) for (int64_t len : {INT64_C(0), INT64_C(1), INT64_C(2), INT64_C(3), most / 2, most - 2, most - 1}) {
        const int64_t off_b = off_a + d;
        const uint32_t from_b = (uint32_t)(off_b - off_a) * 8u;
        uint32_t tail_b = from_b;
        tail_b += (uint32_t)len * 8u;      // (each record adds 8)
        const bool right = (uint64_t)from_b == (uint64_t)d * 8u && (uint64_t)tail_b == (uint64_t)(d + len) * 8u;
        if (il::one_row_counts(off_a, off_b, len) != right) { printf("%lld %lld %lld\n", (long long)off_a, (long long)off_b, (long long)len); return 1; }
    }
    if (il::one_row_counts(2, 0, 5)) return 1;      // (the tail of a stream that lies before the first one would be negative)
    return 0;
}
"""


def test_tails_of_two_streams_of_a_row(tmp_path):
    src = tmp_path / "rules.cpp"
    src.write_text(PROGRAM)
    exe = tmp_path / "rules"
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-I" + os.path.join(ROOT, "include"),
                           "-I" + os.path.join(ROOT, "paper_1812_01776_b200", "csrc"), "-I" + os.path.join(cuda, "include"),
                           str(src), "-o", str(exe), "-L" + os.path.join(cuda, "lib64"), "-lcudart"])
    run = subprocess.run([str(exe)], capture_output=True, text=True)
    assert run.returncode == 0, run.stdout


def test_rows_that_a_kernel_rewrites_are_read_by_plain_loads():
    """node_top_kernel turns a row's records into latencies in place where its one-pass form does not hold: no access to the row
    may take the read-only path (__ldg, ld.global.nc, a pointer said to be const and restrict)."""
    text = open(os.path.join(ROOT, "paper_1812_01776_b200", "csrc", "select_kernel.cu")).read()
    kernel = text[text.index("node_top_kernel(const __grid_constant__"):text.index("size_t node_top_smem")]
    assert "lat[i] = l;" in kernel                                       # it does rewrite the row
    for way in ("__ldg(lat", "__ldg(p.records", "ld.global.nc", "__restrict__"):
        assert way not in kernel, way
