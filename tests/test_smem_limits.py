"""The kernels' dynamic shared-memory limits are kept per device (CPU only): csrc/pic_limits.h against fakes of the
two CUDA calls. Each device that a kernel runs on gets the call, a larger size another one, a smaller none; a
failure is returned, and the call made again."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r'''
#include <cstdio>
#include "pic_limits.h"
static int dev = 0, calls = 0, fail = 0;
cudaError_t CUDARTAPI cudaGetDevice(int* d) { *d = dev; return cudaSuccess; }
cudaError_t CUDARTAPI cudaFuncSetAttribute(const void*, cudaFuncAttribute, int) {
    ++calls;
    return fail ? cudaErrorInvalidValue : cudaSuccess;
}
static int a, b;
static void go(int d, const void* k, size_t n) {
    dev = d;
    const int c0 = calls;
    const cudaError_t e = pic::raise_smem_limit(k, n);
    std::printf("%d%c ", calls - c0, e == cudaSuccess ? 'k' : 'f');
}
int main() {
    go(0, &a, 60000);                  // first use: set
    go(0, &a, 60000); go(0, &a, 50000);  // known
    go(1, &a, 60000);                  // another device: set there too
    go(0, &a, 60000); go(1, &a, 60000);
    go(1, &a, 70000); go(0, &a, 70000);  // larger: set on each
    go(0, &b, 60000);                  // another kernel
    fail = 1; go(2, &a, 60000);        // a failure is returned
    fail = 0; go(2, &a, 60000);        // and the call made again
    go(2, &a, 60000);
}
'''


def test_limits_are_per_device(tmp_path):
    src, exe = tmp_path / "limits.cpp", tmp_path / "limits"
    src.write_text(PROGRAM)
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    subprocess.run(["g++", "-std=c++17", "-I" + os.path.join(ROOT, "paper_1608_04601_gb300", "csrc"),
                    "-I" + os.path.join(cuda, "include"), str(src), "-o", str(exe), "-pthread"], check=True)
    out = subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout.split()
    assert out == ["1k", "0k", "0k", "1k", "0k", "0k", "1k", "1k", "1k", "1f", "1k", "0k"]
