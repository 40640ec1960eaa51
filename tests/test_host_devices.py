"""What the library's host code keeps per device, on a fake CUDA runtime.

The objects of the library are linked with a stand-in for the CUDA runtime that
has two devices of different size: SM counts, and CTA pairs that fit at once,
which also differ between the bf16 and the e4m3 GEMM. A program runs blocks on
both devices, then on eight threads that change devices, and checks the grid of
every GEMM launch against its own device and kernel, and the library's count of
its launches, splits of one to many images among them. Nothing touches a GPU.
"""
import os
import shutil
import subprocess

import pytest

from paper_2606_13898_gb300 import build

PROGRAM = r"""
#include <cuda.h>
#include <cuda_runtime_api.h>
#include <atomic>
#include <mutex>
#include <set>
#include <stdio.h>
#include <string.h>
#include <string>
#include <thread>
#include <map>
#include <vector>
#include "hilo.h"

static thread_local int g_dev = 0;
static const int SMS[2] = {152, 120};
static std::map<const void*, std::string> g_names;  // host stub -> mangled kernel name
static std::atomic<int> g_bad{0}, g_gemms{0}, g_launches{0};

static bool is_gemm(const void* f, bool* fp8) {
  auto it = g_names.find(f);
  if (it == g_names.end() || it->second.find("gemm2_kernel") == std::string::npos) return false;
  *fp8 = it->second.find("ILb1E") != std::string::npos;
  return true;
}
static int pairs(int dev, bool fp8) { return SMS[dev] / 2 - (fp8 ? 3 : 0); }

static CUresult encode(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                       const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                       CUtensorMapL2promotion, CUtensorMapFloatOOBfill) { return CUDA_SUCCESS; }

extern "C" {
void** __cudaRegisterFatBinary(void*) { static void* h; return &h; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char* host, char*, const char* name, int, void*, void*, void*, void*, int*) {
  g_names[host] = name;
}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
int __cudaPushCallConfiguration(dim3, dim3, size_t, void*) { return 0; }
int __cudaPopCallConfiguration(dim3*, dim3*, size_t*, void*) { return 0; }
int __cudaGetKernel(void**, const void*) { return 0; }
int __cudaLaunchKernel(void*, dim3, dim3, void**, size_t, void*) { return 0; }
cudaError_t cudaGetDevice(int* d) { *d = g_dev; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr a, int d) {
  *v = a == cudaDevAttrComputeCapabilityMajor ? 10 : a == cudaDevAttrComputeCapabilityMinor ? 3 : SMS[d];
  return cudaSuccess;
}
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaFuncGetAttributes(cudaFuncAttributes* a, const void*) {
  memset(a, 0, sizeof(*a));
  a->numRegs = 168;
  return cudaSuccess;
}
cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaGetDriverEntryPointByVersion(const char*, void** p, unsigned, unsigned long long,
                                             cudaDriverEntryPointQueryResult* q) {
  *p = reinterpret_cast<void*>(&encode);
  *q = cudaDriverEntryPointSuccess;
  return cudaSuccess;
}
const char* cudaGetErrorString(cudaError_t) { return "fake"; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaGetSymbolAddress(void** p, const void*) { *p = nullptr; return cudaErrorInvalidValue; }
cudaError_t cudaMemcpyFromSymbol(void* d, const void*, size_t n, size_t, cudaMemcpyKind) { memset(d, 0, n); return cudaSuccess; }
cudaError_t cudaMemcpyToSymbol(const void*, const void*, size_t, size_t, cudaMemcpyKind) { return cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveClusters(int* n, const void* f, const cudaLaunchConfig_t*) {
  bool fp8;
  if (!is_gemm(f, &fp8)) return cudaErrorInvalidValue;
  std::this_thread::yield();  // let other threads' first calls in
  *n = pairs(g_dev, fp8);
  return cudaSuccess;
}
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* f, void**) {
  bool fp8;
  ++g_launches;
  if (is_gemm(f, &fp8)) {
    ++g_gemms;
    if (static_cast<int>(c->gridDim.x) != 2 * pairs(g_dev, fp8)) {
      if (!g_bad++) printf("device %d, %s: grid %u, want %d\n", g_dev, fp8 ? "e4m3" : "bf16", c->gridDim.x, 2 * pairs(g_dev, fp8));
    }
  }
  return cudaSuccess;
}
}

static int block(bool fp8) {
  static char mem[64] __attribute__((aligned(256)));  // never read: every launch is a fake
  hilo_shape s = {1, 8, 8, 1024, 4, 8, 1, 1, 0};
  hilo_block_weights w;
  hilo_block_weights_fp8 w8;
  for (size_t i = 0; i < sizeof(w) / sizeof(void*); ++i) reinterpret_cast<void**>(&w)[i] = mem;
  for (size_t i = 0; i < sizeof(w8) / sizeof(void*); ++i) reinterpret_cast<void**>(&w8)[i] = mem;
  const size_t big = size_t{1} << 40;
  return fp8 ? hilo_block_forward_fp8(&s, &w8, reinterpret_cast<int*>(mem), 64, mem, mem, HILO_BF16,
                                      reinterpret_cast<float*>(mem), mem, big, nullptr)
             : hilo_block_forward(&s, &w, reinterpret_cast<int*>(mem), 64, mem, mem, HILO_BF16,
                                  reinterpret_cast<float*>(mem), mem, big, nullptr);
}

static int split(int B) {
  static char mem[64] __attribute__((aligned(256)));
  hilo_shape s = {B, 8, 8, 1024, 0, 8, 1, 1, 0};
  int* p = reinterpret_cast<int*>(mem);
  hilo_split_out o = {reinterpret_cast<uint8_t*>(mem), p, p, p, p};
  return hilo_split(&s, reinterpret_cast<float*>(mem), reinterpret_cast<uint8_t*>(mem), p, p, &o, nullptr, 0, nullptr);
}

int main(int argc, char** argv) {
  auto run = [](int first, int n) {
    for (int i = 0; i < n; ++i) {
      g_dev = (first + i / 2) % 2;
      const int rc = block((first + i) % 2) | split(1 + i);
      if (rc != HILO_OK) {
        printf("block: %d (%s)\n", rc, hilo_last_error());
        ++g_bad;
        return;
      }
    }
  };
  if (argc > 1 && !strcmp(argv[1], "threads")) {
    std::vector<std::thread> ts;
    for (int t = 0; t < 8; ++t) ts.emplace_back(run, t, 40);
    for (auto& t : ts) t.join();
  } else {
    run(0, 20);
  }
  if (hilo_launch_count() != static_cast<unsigned long long>(g_launches)) {
    printf("hilo_launch_count %llu of %d launches\n", hilo_launch_count(), g_launches.load());
    ++g_bad;
  }
  printf("%d GEMM launches, %d bad\n", g_gemms.load(), g_bad.load());
  return g_bad || !g_gemms;
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("g++ not found")
    build.build()
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(build._nvcc()))), "include")
    d = tmp_path_factory.mktemp("devices")
    src, exe = d / "devices.cpp", d / "devices"
    src.write_text(PROGRAM)
    objs = [os.path.join(build.BUILD, s.replace(".cu", ".o")) for s in build.SOURCES]
    r = subprocess.run([gxx, "-std=c++17", "-O1", "-I", cuda, "-I", build.INCLUDE, "-o", str(exe), str(src), *objs,
                        "-lpthread"], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-3000:]
    return str(exe)


@pytest.mark.parametrize("how", ["one thread", "threads"])
def test_gemm_grids_follow_their_device_and_kernel(program, how):
    r = subprocess.run([program, how], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout + r.stderr
