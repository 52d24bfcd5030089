"""Function attributes (dynamic shared memory, non-portable cluster sizes) and what fits belong to a
device: the seeding's host code asks on each device it runs on.  The host part of the k-means object
is linked against a stand-in for the CUDA runtime that keeps attributes per device, as CUDA does."""
import os
import subprocess

from paper_2307_00071_gb300 import build_lib

MAIN = r"""
#include <cstdint>
#include <cstdio>
#include <map>
#include <utility>
#include <cuda_runtime_api.h>

namespace gira {   // of gira_internal.cuh
struct DeviceState;
int kpp_cluster_size(int64_t n);
cudaError_t launch_kpp_cluster(const float4*, int64_t n, int k, uint64_t, float4*, int64_t*, int cs, DeviceState*,
                               cudaStream_t);
int kpp_blocks_per_warp(int64_t n, int dim);
cudaError_t launch_kpp_blocks(const float4*, int64_t n, int k, uint64_t, float4*, int64_t*, float*, int nsb,
                              DeviceState*, cudaStream_t, int dim);
}

static int device = 0;
static std::map<std::pair<int, const void*>, int> smem, wide;   // (device, function) -> attribute
extern "C" {
cudaError_t cudaGetDevice(int* d) { *d = device; return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) { *v = 152; return cudaSuccess; }
cudaError_t cudaFuncSetAttribute(const void* f, cudaFuncAttribute a, int v) {
    (a == cudaFuncAttributeMaxDynamicSharedMemorySize ? smem : wide)[{device, f}] = v;
    return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveClusters(int* n, const void* f, const cudaLaunchConfig_t* c) {
    const int cs = (int)c->attrs[0].val.clusterDim.x;
    *n = device != 2 && smem[{device, f}] >= (int)c->dynamicSmemBytes && (cs <= 8 || wide[{device, f}]);
    return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void*, int, size_t, unsigned) {
    *n = 1;
    return cudaSuccess;
}
cudaError_t cudaLaunchCooperativeKernel(const void*, dim3, dim3, void**, size_t, cudaStream_t) { return cudaSuccess; }
// refused as CUDA does: more shared memory or a wider cluster than the device's attributes allow
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* f, void**) {
    if ((int)c->dynamicSmemBytes > 48 * 1024 && smem[{device, f}] < (int)c->dynamicSmemBytes) return cudaErrorInvalidValue;
    if (c->attrs[0].val.clusterDim.x > 8 && !wide[{device, f}]) return cudaErrorInvalidClusterSize;
    return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t, dim3, dim3, void**, size_t, cudaStream_t) { return cudaSuccess; }
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* f) { *k = (cudaKernel_t)f; return cudaSuccess; }
unsigned __cudaPushCallConfiguration(dim3, dim3, size_t, void*) { return 0; }
cudaError_t __cudaPopCallConfiguration(dim3*, dim3*, size_t*, void*) { return cudaSuccess; }
void** __cudaRegisterFatBinary(void*) { static void* h; return &h; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char*, char*, const char*, int, void*, void*, void*, void*, int*) {}
}

int main() {
    using namespace gira;
    for (int d : {0, 1, 2, 1, 0}) {
        device = d;
        const int cs = kpp_cluster_size(1000), nsb3 = kpp_blocks_per_warp(300000, 3), nsb4 = kpp_blocks_per_warp(300000, 4);
        const bool one = cs && launch_kpp_cluster(nullptr, 1000, 2, 0, nullptr, nullptr, cs, nullptr, nullptr) == cudaSuccess;
        const bool l3 = nsb3 && launch_kpp_blocks(nullptr, 300000, 2, 0, nullptr, nullptr, nullptr, nsb3, nullptr, nullptr, 3) == cudaSuccess;
        const bool l4 = nsb4 && launch_kpp_blocks(nullptr, 300000, 2, 0, nullptr, nullptr, nullptr, nsb4, nullptr, nullptr, 4) == cudaSuccess;
        std::printf("%d: %d %d %d\n", d, one, l3, l4);
    }
    return 0;
}
"""


def test_seeding_asks_on_every_device(tmp_path):
    build_lib.build()
    src, exe = tmp_path / "main.cpp", tmp_path / "main"
    src.write_text(MAIN)
    cuda = os.path.join(os.path.dirname(os.path.dirname(build_lib.NVCC)), "include")
    subprocess.run(["g++", "-std=c++17", "-no-pie", "-I", cuda, str(src),
                    os.path.join(build_lib.OUT_DIR, "kmeans_kernels.o"), "-o", str(exe)], check=True)
    got = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout
    runs = "1 1 1"
    assert got.splitlines() == [f"0: {runs}", f"1: {runs}", "2: 0 0 0", f"1: {runs}", f"0: {runs}"]
