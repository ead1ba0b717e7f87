"""The opt-in to more than 48 KB of dynamic shared memory reaches every device a kernel is
launched on, not only the process's first. The helper is compiled against a fake runtime of
three devices that refuses a launch without the opt-in on the current one."""
import glob
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2407_07096_gb300", "csrc")

MAIN = r"""
#include "smem_opt_in.h"
#include <stdio.h>
static int g_dev = 0, g_calls = 0, g_limit[3][2];  // per device and kernel, as the driver keeps it
static char g_kernels[2];
static bool g_fail = false;
extern "C" cudaError_t cudaGetDevice(int *d) { *d = g_dev; return cudaSuccess; }
extern "C" cudaError_t cudaFuncSetAttribute(const void *f, cudaFuncAttribute, int v) {
    ++g_calls;
    if (g_fail) return cudaErrorInvalidValue;
    g_limit[g_dev][(const char *)f - g_kernels] = v;
    return cudaSuccess;
}
static stagkde::SmemOptIn g_in[2];
static bool launch(int k, int bytes) {
    if (g_in[k](g_kernels + k, bytes) != cudaSuccess) return false;
    return bytes <= 49152 || g_limit[g_dev][k] >= bytes;
}
int main() {
    int bad = 0;
    for (int round = 0; round < 2; ++round)
        for (g_dev = 0; g_dev < 3; ++g_dev)
            for (int k = 0; k < 2; ++k) bad += !launch(k, 55296 + k);
    if (g_calls != 6) bad += 100;  // once per device and kernel
    g_fail = true;
    stagkde::SmemOptIn again;
    g_dev = 1;
    if (again(g_kernels, 60000) != cudaErrorInvalidValue) bad += 1000;
    g_fail = false;
    if (again(g_kernels, 60000) != cudaSuccess || g_limit[1][0] != 60000) bad += 10000;  // a failure is not kept
    printf("%d\n", bad);
    return bad != 0;
}
"""


def test_every_device_is_opted_in(tmp_path):
    src = tmp_path / "main.cpp"
    src.write_text(MAIN)
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    exe = str(tmp_path / "main")
    subprocess.run(["g++", "-std=c++17", "-O1", f"-I{CSRC}", f"-I{cuda}/include", "-o", exe, str(src)], check=True)
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout


def test_no_launch_opts_in_by_itself():
    for path in glob.glob(os.path.join(CSRC, "*.c*")):
        with open(path) as f:
            assert "cudaFuncSetAttribute" not in f.read(), path
