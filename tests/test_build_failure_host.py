"""A build whose launch fails part way (host check, no GPU): the library's objects are linked with a
stand-in for the CUDA runtime whose launches do nothing but keep the selection's accumulators as the
kernels would, and which can fail the n-th launch.  After a failed build the next one on the same
handle, and on the static scratch, has to find the accumulators at zero."""
import glob
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
PKG = os.path.join(ROOT, "paper_2004_05188_gb300")

RUNTIME = r"""
#include <cstdlib>
#include <cstring>
#include <map>
#include <string>
#include <cuda_runtime_api.h>

static std::map<const void*, std::string> g_name;

extern "C" {
int g_fail = 0, g_capturing = 0;
void on_launch(const char* name, void** args);

void** __cudaRegisterFatBinary(void*) { static void* h; return &h; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
void __cudaRegisterFunction(void**, const char* fun, char*, const char* name, int, uint3*, uint3*, dim3*, dim3*, int*) {
  g_name[fun] = name;
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t*, const void* f, void** args) {
  if (g_fail > 0 && --g_fail == 0) return cudaErrorLaunchOutOfResources;
  if (!g_capturing) on_launch(g_name[f].c_str(), args);  // (a captured launch does not run)
  return cudaSuccess;
}
cudaError_t cudaMalloc(void** p, size_t n) { *p = aligned_alloc(256, (n + 255) / 256 * 256); return cudaSuccess; }
cudaError_t cudaFree(void* p) { free(p); return cudaSuccess; }
cudaError_t cudaMemset(void* p, int v, size_t n) { memset(p, v, n); return cudaSuccess; }
cudaError_t cudaMemsetAsync(void* p, int v, size_t n, cudaStream_t) {
  if (!g_capturing) memset(p, v, n);
  return cudaSuccess;
}
cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus* s) {
  *s = g_capturing ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone;
  return cudaSuccess;
}
cudaError_t cudaGetDevice(int* d) { *d = 0; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr a, int) {
  *v = a == cudaDevAttrMultiProcessorCount ? 4 : 232448;
  return cudaSuccess;
}
cudaError_t cudaDeviceSynchronize(void) { return cudaSuccess; }
cudaError_t cudaGetLastError(void) { return cudaSuccess; }
const char* cudaGetErrorString(cudaError_t) { return "stand-in"; }
cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessor(int* n, const void*, int, size_t) { *n = 1; return cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void*, int, size_t, unsigned) {
  *n = 1;
  return cudaSuccess;
}
cudaError_t cudaGetSymbolAddress(void** p, const void*) {
  static void* scratch = calloc(1, 64 << 20);
  *p = scratch;
  return cudaSuccess;
}
}
"""

HARNESS = r"""
#include <cstdio>
#include <cstring>
#include "ps.h"
#include "ps_internal.cuh"

static int g_stale = 0, g_selects = 0;
extern "C" {
extern int g_fail, g_capturing;
void on_launch(const char* name, void** args) {
  if (strstr(name, "k_select_bbox")) {
    ps::Geo* geo = *static_cast<ps::Geo**>(args[6]);
    ++g_selects;
    g_stale += geo->acc_sel != 0 || geo->acc_status != 0;
    for (uint32_t b : geo->acc_box) g_stale += b != 0;
    geo->acc_sel += (uint32_t)*static_cast<int64_t*>(args[2]);
    for (uint32_t& b : geo->acc_box) b = 7;
    geo->acc_status = 2;
  } else if (strstr(name, "k_count")) {
    ps::Geo* geo = *static_cast<ps::Geo**>(args[2]);
    geo->acc_sel = 0, geo->acc_status = 0;
    for (uint32_t& b : geo->acc_box) b = 0;
  }
}
}

int main() {
  alignas(16) static float xyz[300];
  alignas(16) static uint8_t type[100];
  uint64_t all[4] = {~0ull, ~0ull, ~0ull, ~0ull}, rdf[10], meta[16];
  int bad = 0;
  ps_grid* g = nullptr;
  if (ps_grid_create(100, nullptr, &g)) return puts("create failed"), 1;
  for (int at = 1; at <= 5; ++at)
    for (int captured = 0; captured < 2; ++captured) {
      g_fail = at;  // the at-th launch of the build fails
      if (ps_grid_build(g, xyz, type, 100, all, 1.0f, nullptr) != PS_ERR_CUDA) printf("build %d did not fail\n", at), ++bad;
      g_fail = 0;
      if (captured) {  // a build that is recorded for later does not run
        g_capturing = 1;
        if (ps_grid_build(g, xyz, type, 100, all, 1.0f, nullptr) != PS_OK) printf("captured build %d\n", at), ++bad;
        g_capturing = 0;
      }
      for (int k = 0; k < 2; ++k)
        if (ps_grid_build(g, xyz, type, 100, all, 1.0f, nullptr) != PS_OK) printf("build after %d\n", at), ++bad;
      if (g_stale) printf("handle, launch %d failed: stale accumulators\n", at), ++bad, g_stale = 0;
    }
  ps_grid_destroy(g);
  const ps_bins bins = {0.0, 0.1, 10};
  auto call = [&]() {
    return ps_spatstat_static(xyz, type, nullptr, 100, all, 1.0f, all, 0.0f, bins, nullptr, 0, rdf, nullptr, meta, nullptr,
                              nullptr, nullptr);
  };
  for (int at = 1; at <= 5; ++at) {
    g_fail = at;
    if (call() != PS_ERR_CUDA) printf("static call %d did not fail\n", at), ++bad;
    g_fail = 0;
    for (int k = 0; k < 2; ++k)
      if (call() != PS_OK) printf("static call after %d: %s\n", at, ps_last_error()), ++bad;
    if (g_stale) printf("static scratch, launch %d failed: stale accumulators\n", at), ++bad, g_stale = 0;
  }
  if (g_selects < 30) printf("%d selections seen\n", g_selects), ++bad;
  printf(bad ? "FAIL %d\n" : "OK\n", bad);
  return bad ? 1 : 0;
}
"""


def test_accumulators_after_a_failed_build(tmp_path):
    nvcc = shutil.which("nvcc") or ("/usr/local/cuda/bin/nvcc" if os.path.exists("/usr/local/cuda/bin/nvcc") else None)
    if nvcc is None:
        pytest.skip("nvcc not found")
    from paper_2004_05188_gb300 import _build

    _build.build()
    want = [os.path.join(_build.BUILD, os.path.basename(s) + ".o") for s in glob.glob(os.path.join(PKG, "csrc", "*.cu"))]
    if not all(os.path.exists(o) for o in want):
        _build.build(force=True)
    src, rt = tmp_path / "build.cu", tmp_path / "runtime.cpp"
    src.write_text(HARNESS)
    rt.write_text(RUNTIME)
    exe = tmp_path / "build"
    subprocess.check_call([nvcc, "-std=c++17", "-cudart", "none", "-I", os.path.join(PKG, "csrc"), "-I",
                           os.path.join(ROOT, "include"), "-Xlinker", "--unresolved-symbols=ignore-all", "-o", str(exe),
                           str(src), str(rt), *sorted(want)])
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0 and r.stdout.strip().endswith("OK"), r.stdout + r.stderr
