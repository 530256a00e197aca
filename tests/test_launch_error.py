"""A launch that fails is reported by its own call and leaves no error behind
for the next one. launch_after runs on the host against a runtime of this
file's own that refuses as the real one does: it returns the error and keeps
it as the last error until cudaGetLastError takes it."""
import subprocess

from paper_2607_20214_gb300 import build

RUNTIME = r"""
#include <cuda_runtime_api.h>
cudaError_t last = cudaSuccess;
bool refuse_smem = false, refuse_launch = false;
int launches = 0;
static cudaError_t refuse(bool no, cudaError_t e) {
    if (no) last = e;
    return no ? e : cudaSuccess;
}
extern "C" {
cudaError_t cudaGetLastError() {
    const cudaError_t e = last;
    last = cudaSuccess;
    return e;
}
cudaError_t cudaFuncSetAttribute(const void *, cudaFuncAttribute, int) {
    return refuse(refuse_smem, cudaErrorInvalidValue);
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t *, const void *,
                                void **) {
    ++launches;
    return refuse(refuse_launch, cudaErrorInvalidConfiguration);
}
// what the compiler's start-up code asks for
static void *module;
void **__cudaRegisterFatBinary(void *) { return &module; }
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **) {}
char __cudaInitModule(void **) { return 0; }
}
"""

CALLS = r"""
#include <stdio.h>
#include "device_common.cuh"

extern cudaError_t last;
extern bool refuse_smem, refuse_launch;
extern int launches;
static void nothing(int) {}

int main() {
    auto launch = [](size_t smem) {
        return elsaa::launch_after(nothing, dim3(1), 32, smem, nullptr, 1);
    };
    int bad = 0;
    auto expect = [&](const char *what, bool ok) {
        if (!ok) printf("not so: %s\n", what);
        bad += !ok;
    };
    expect("a launch succeeds", launch(0) == cudaSuccess);
    refuse_launch = true;
    expect("a refused launch returns its error",
           launch(1 << 16) == cudaErrorInvalidConfiguration);
    expect("it leaves none behind", last == cudaSuccess);
    refuse_launch = false;
    refuse_smem = true;
    const int n = launches;
    expect("refused shared memory returns its error",
           launch(1 << 20) == cudaErrorInvalidValue);
    expect("nothing is launched", launches == n);
    expect("no error is left behind", last == cudaSuccess);
    return bad;
}
"""


def test_a_failed_launch_leaves_no_error(tmp_path):
    files = []
    for name, text in (("runtime.cpp", RUNTIME), ("calls.cu", CALLS)):
        files.append(str(tmp_path / name))
        with open(files[-1], "w") as f:
            f.write(text)
    exe = str(tmp_path / "calls")
    subprocess.run([build.nvcc(), *build.ARCH, *build.NVCC_FLAGS, "-I",
                    build.CSRC, "-cudart", "none", *files, "-o", exe],
                   check=True, capture_output=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout + r.stderr
