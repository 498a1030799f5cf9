"""The opt-in to dynamic shared memory and the resident-CTA count of a kernel
(csrc/resident.h) against a stand-in for the CUDA runtime: asked for once on
every device, not once per process, and again after a failure."""
import os
import re
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2104_08571_gb300", "csrc")

RUNTIME = """
#pragma once
#include <cstddef>
enum cudaError_t { cudaSuccess = 0, cudaErrorUnknown = 999 };
enum cudaFuncAttribute { cudaFuncAttributeMaxDynamicSharedMemorySize = 8 };
extern int g_device, g_smem[128], g_sets, g_fail, g_cleared;
inline cudaError_t cudaGetDevice(int* d) { *d = g_device; return cudaSuccess; }
inline cudaError_t cudaGetLastError() { ++g_cleared; return cudaSuccess; }
template <class K>
cudaError_t cudaFuncSetAttribute(K, cudaFuncAttribute, int v)
{
    ++g_sets;
    if (g_fail == 1) return cudaErrorUnknown;
    g_smem[g_device] = v;
    return cudaSuccess;
}
template <class K>
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessor(int* n, K, int threads, size_t smem)
{
    *n = g_fail == 2 ? 7 : (int)(1000 * g_device + threads + smem);
    return g_fail == 2 ? cudaErrorUnknown : cudaSuccess;
}
"""

PROGRAM = """
#include "resident.h"
#include <cassert>
#include <initializer_list>
int g_device, g_smem[128], g_sets, g_fail, g_cleared;
static void kern() {}
int main()
{
    ripple::ResidentCtas r;
    for (int pass = 0; pass < 3; ++pass)
        for (int d : {0, 3, 1}) {
            g_device = d;
            assert(r.get(kern, 10, 200) == 1000 * d + 210);
            assert(g_smem[d] == 200);
        }
    assert(g_sets == 3);  // once per device
    for (int pass = 0; pass < 2; ++pass) {  // a device number beyond the table: asked for every time
        g_device = 100;
        assert(r.get(kern, 10, 200) == 100210);
    }
    assert(g_sets == 5);
    g_device = 2;
    for (g_fail = 1; g_fail <= 2; ++g_fail) assert(r.get(kern, 10, 200) == 0);
    assert(g_cleared == 2);
    g_fail = 0;
    assert(r.get(kern, 10, 200) == 2210 && g_smem[2] == 200);  // a failure is not kept
    g_fail = 1;
    assert(r.get(kern, 10, 200) == 2210);
    return 0;
}
"""


@pytest.mark.skipif(not shutil.which("g++"), reason="no C++ compiler")
def test_opt_in_per_device_and_after_a_failure(tmp_path):
    (tmp_path / "cuda_runtime.h").write_text(RUNTIME)
    (tmp_path / "main.cpp").write_text(PROGRAM)
    exe = str(tmp_path / "t")
    subprocess.run(["g++", "-std=c++17", "-UNDEBUG", "-I", str(tmp_path), "-I", CSRC, str(tmp_path / "main.cpp"), "-o", exe],
                   check=True)
    subprocess.run([exe], check=True)


def test_no_opt_in_is_kept_per_process():
    """No function-local static holds the outcome of a per-device runtime call."""
    for name in sorted(os.listdir(CSRC)):
        text = open(os.path.join(CSRC, name)).read()
        assert not re.search(r"static (const )?(int|bool) \w+(\[\d\])? = (\[|false|\{false)", text), name
