"""What a launch sets once (a kernel's dynamic shared memory limit) belongs to a
device: a process that uses a second GPU sets it there too.  Checked without a
GPU: the launch code (warpseg.cu, which holds no kernel) is compiled against a
fake CUDA runtime with two devices, which records the attributes set on each."""
import os
import subprocess

from paper_2607_14054_gb300 import buildlib

# two devices; a launch above 48 KB of shared memory needs the attribute on its device
RUNTIME = r"""
#include <map>
#include <utility>
#include <cuda_runtime_api.h>

int g_dev = 0, g_failed = 0;
static std::map<std::pair<int, const void*>, int> g_limit;
extern "C" {
cudaError_t cudaGetDevice(int* d) { *d = g_dev; return cudaSuccess; }
cudaError_t cudaFuncSetAttribute(const void* f, cudaFuncAttribute a, int v) {
    if (a == cudaFuncAttributeMaxDynamicSharedMemorySize) g_limit[{g_dev, f}] = v;
    return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessor(int* n, const void* f, int, size_t s) {
    *n = (size_t)g_limit[{g_dev, f}] >= s || s <= 49152 ? 2 + g_dev : 0;
    return cudaSuccess;
}
static cudaError_t launch(const void* f, size_t smem) {
    if (smem > 49152 && (size_t)g_limit[{g_dev, f}] < smem) {
        ++g_failed;
        return cudaErrorInvalidValue;
    }
    return cudaSuccess;
}
cudaError_t cudaLaunchKernel(const void* f, dim3, dim3, void**, size_t smem, cudaStream_t) {
    return launch(f, smem);
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* f, void**) {
    return launch(f, c->dynamicSmemBytes);
}
void** __cudaRegisterFatBinary(void*) { return nullptr; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
char __cudaInitModule(void**) { return 0; }
}

"""

MAIN = r"""
#include <cstdio>
#include "sos_common.cuh"

extern int g_dev, g_failed;

namespace sosf {
static int k[9];
const void* warpseg_fn_16(bool cr) { return &k[cr]; }
const void* warpseg_fn_32(bool cr) { return &k[2 + cr]; }
const void* warpseg_fn_64(bool cr) { return &k[4 + cr]; }
const void* stream_fn_16() { return &k[6]; }
const void* stream_fn_32() { return &k[7]; }
const void* stream_fn_64() { return &k[8]; }
cudaError_t launch_warpseg(const Params& p, int64_t grid, cudaStream_t stream, bool early);
cudaError_t launch_stream(const Params& p, int64_t chunk, int64_t seg_len, int32_t maxseg,
                          int32_t foreign, cudaStream_t stream);
int warpseg_ctas_per_sm(int N, int algo, int dev);
}

int main() {
    for (int round = 0; round < 2; ++round)
        for (g_dev = 0; g_dev < 2; ++g_dev)
            for (int N = 16; N <= 64; N *= 2) {
                sosf::Params p{};
                p.N = N;
                p.C = 1;
                p.dev = sosf::device_slot();
                for (int algo = 1; algo <= 2; ++algo) {
                    p.algo = algo;
                    if (sosf::warpseg_ctas_per_sm(N, algo, g_dev) != 2 + g_dev) ++g_failed;
                    if (sosf::launch_warpseg(p, 4, nullptr, true) != cudaSuccess) ++g_failed;
                }
                if (sosf::launch_stream(p, 100, 100, 1, 0, nullptr) != cudaSuccess) ++g_failed;
            }
    std::printf("%d\n", g_failed);
    return g_failed != 0;
}
"""


def test_second_device_is_set_up(tmp_path):
    runtime, main, exe = tmp_path / "runtime.cpp", tmp_path / "main.cu", tmp_path / "check"
    runtime.write_text(RUNTIME)
    main.write_text(MAIN)
    inc = ["-I", buildlib.CSRC, "-I", os.path.dirname(buildlib.INCLUDE)]
    subprocess.run([buildlib._nvcc(), "-gencode", "arch=compute_103a,code=sm_103a", "-std=c++17",
                    "-cudart", "none", *inc, "-o", str(exe), str(runtime), str(main),
                    os.path.join(buildlib.CSRC, "warpseg.cu")], check=True)
    r = subprocess.run([str(exe)], stdout=subprocess.PIPE, timeout=60)
    assert r.returncode == 0, r.stdout
