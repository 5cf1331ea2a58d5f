"""CPU test of the kept occupancy answers: the header that the launchers
include, compiled with the host compiler against a driver of its own."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

HARNESS = r"""
#include <cuda_runtime.h>
#include "htex_internal.h"

static int answers = 0, asked = 0, status = 0;

extern "C" cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessor(int* b, const void*, int, size_t) {
    ++asked;
    *b = answers;
    return status ? cudaErrorUnknown : cudaSuccess;
}
extern "C" cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* b, const void* k, int t, size_t s, unsigned) {
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(b, k, t, s);
}
extern "C" cudaError_t cudaGetLastError() { return cudaSuccess; }

static void kernel() {}

int main() {
    static Occupancy o;
    status = 1, answers = 7;
    if (o.get(kernel, 256, 0) != 1) return 1;                    // the driver failed: one block, for now
    status = 0, answers = 5;
    if (o.get(kernel, 256, 0) != 5 || asked != 2) return 2;      // asked again
    answers = 9;
    if (o.get(kernel, 256, 0) != 5 || asked != 2) return 3;      // kept
    if (o.get(kernel, 256, 1) != 9 || asked != 3) return 4;      // per device
    if (o.get(kernel, 256, 64) != 9 || o.get(kernel, 256, -1) != 9 || asked != 5) return 5;   // not kept past the table
    answers = 0;
    if (o.get(kernel, 256, 2) != 1) return 6;
    answers = 3;
    if (o.get(kernel, 256, 2) != 3) return 7;
    return 0;
}
"""


def test_only_the_drivers_answers_are_kept(tmp_path):
    """A query that fails gives one block and is asked again; an answer is
    kept per device."""
    src, exe = tmp_path / "occupancy.cpp", tmp_path / "occupancy"
    src.write_text(HARNESS)
    cuda = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include")
    subprocess.run(["g++", "-O1", "-std=c++17", "-I", os.path.join(ROOT, "include"), "-I",
                    os.path.join(ROOT, "paper_2207_05618_gb300", "csrc"), "-I", cuda, str(src), "-o", str(exe)], check=True)
    assert subprocess.run([str(exe)]).returncode == 0
