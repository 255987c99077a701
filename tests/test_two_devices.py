"""The convolution launchers on two devices of one process, from two host threads: the compiled launch code
linked against a stand-in for the CUDA runtime that keeps the shared-memory opt-in per kernel AND device, as the
runtime does, and refuses a launch above 48 KB without it."""
import glob
import os
import shutil
import subprocess

import pytest

from paper_1705_08849_gb300 import build

MAIN = r"""
#include <cstddef>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <map>
#include <mutex>
#include <thread>
#include <utility>
#include <vector>

#include "fit.h"

struct dim3 { unsigned x, y, z; };
struct Config { dim3 grid, block; size_t smem; void* stream; };
static std::mutex mu;
static thread_local int device = 0;
static thread_local int error = 0;
static thread_local std::vector<Config> configs;
static thread_local dim3 last_grid;
static std::map<std::pair<const void*, int>, int> optin;
static std::map<std::pair<const void*, int>, int> queries;
static int launches = 0;
static const int kSms[2] = {100, 40};

extern "C" {
void** __cudaRegisterFatBinary(void*) { static void* h; return &h; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction() {}
void __cudaRegisterVar() {}
int __cudaGetKernel(const void** k, const void* f) { *k = f; return 0; }
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t m, void* s) { configs.push_back({g, b, m, s}); return 0; }
int __cudaPopCallConfiguration(dim3* g, dim3* b, size_t* m, void* s) {
  const Config c = configs.back();
  configs.pop_back();
  *g = c.grid, *b = c.block, *m = c.smem, *(void**)s = c.stream;
  return 0;
}
int __cudaLaunchKernel(const void* k, dim3 g, dim3, void**, size_t smem, void*) {
  std::lock_guard<std::mutex> lock(mu);
  auto it = optin.find({k, device});
  if (smem > 48 * 1024 && (it == optin.end() || (size_t)it->second < smem)) return error = 1;
  last_grid = g;
  ++launches;
  return 0;
}
int cudaGetLastError() { const int e = error; error = 0; return e; }
const char* cudaGetErrorString(int e) { return e ? "invalid argument" : "no error"; }
int cudaGetDevice(int* d) { *d = device; return 0; }
int cudaSetDevice(int d) { device = d; return 0; }
int cudaDeviceGetAttribute(int* v, int attr, int d) {
  *v = attr == 16 ? kSms[d] : 228 * 1024;  // 16: SM count; else the SM's shared memory
  return 0;
}
int cudaFuncSetAttribute(const void* f, int, int v) {
  std::lock_guard<std::mutex> lock(mu);
  optin[{f, device}] = v;
  return 0;
}
int cudaFuncGetAttributes(void* a, const void*) {
  int* w = (int*)a;  // (three size_t, two int, then numRegs are what matters)
  std::memset(a, 0, 56);
  for (int i = 6; i < 10; ++i) w[i] = 64;
  return 0;
}
int cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void* f, int, size_t, unsigned) {
  std::lock_guard<std::mutex> lock(mu);
  ++queries[{f, device}];
  *n = 3 - device;
  return 0;
}
int cudaMemsetAsync(void*, int, size_t, void*) { return 0; }
int cudaMallocAsync(void** p, size_t, void*) { *p = (void*)256; return 0; }
int cudaFreeAsync(void*, void*) { return 0; }
static int encode_tiled() { return 0; }
int cudaGetDriverEntryPointByVersion(const char*, void** fn, unsigned, unsigned long long, int* q) {
  *fn = (void*)encode_tiled;
  *q = 0;
  return 0;
}
}

static int failures = 0;
static void expect(bool ok, const char* what, int dev, int a, int b) {
  if (ok) return;
  std::lock_guard<std::mutex> lock(mu);
  ++failures;
  std::printf("device %d, %d -> %d: %s (%s)\n", dev, a, b, what, fit_last_error());
}

static void all_layers(int dev) {
  cudaSetDevice(dev);
  static const int shapes[][2] = {{16, 16}, {16, 32}, {32, 32}, {32, 64}, {64, 64}, {64, 32}, {32, 16}};
  void* p = (void*)4096;
  for (auto& s : shapes) {
    const int a = s[0], b = s[1], n = 64;
    expect(fit_unet_conv3_wgrad(n, n, n, a, b, p, p, (float*)p, (float*)p, nullptr) == FIT_OK, "weight gradient", dev, a, b);
    // one wave: a third of the device's resident blocks for each of the three z-taps
    expect(last_grid.x == (unsigned)((3 - dev) * kSms[dev] / 3) && last_grid.y == 3, "weight-gradient grid", dev, a, b);
    expect(fit_unet_conv3(n, n, n, a, b, p, (float*)p, (float*)p, 1, p, nullptr) == FIT_OK, "conv", dev, a, b);
    expect(fit_unet_conv3_dgrad(n, n, n, a, b, p, (float*)p, p, nullptr) == FIT_OK, "data gradient", dev, a, b);
  }
  expect(fit_unet_tconv(32, 32, 32, 64, 32, p, (float*)p, (float*)p, p, nullptr) == FIT_OK, "transposed conv", dev, 64, 32);
  expect(fit_unet_tconv(32, 32, 32, 32, 16, p, (float*)p, (float*)p, p, nullptr) == FIT_OK, "transposed conv", dev, 32, 16);
}

int main(int argc, char** argv) {
  const bool threads = argc > 1 && !std::strcmp(argv[1], "threads");
  if (threads) {
    std::thread t[8];
    for (int i = 0; i < 8; ++i) t[i] = std::thread(all_layers, i % 2);
    for (auto& x : t) x.join();
  } else {
    for (int dev : {0, 1, 0}) all_layers(dev);
  }
  for (auto& q : queries) expect(q.second == 1, "occupancy asked more than once", q.first.second, q.second, 0);
  expect(launches > 0, "nothing launched", 0, 0, 0);
  return failures != 0;
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    if shutil.which("g++") is None:
        pytest.skip("needs g++")
    build.build()
    d = tmp_path_factory.mktemp("two_devices")
    src, exe = d / "main.cpp", d / "main"
    src.write_text(MAIN)
    objs = sorted(glob.glob(os.path.join(build.BUILD, "fit_*.o")))
    # what the launches under test never call stays unresolved
    subprocess.run(["g++", "-std=c++17", "-O1", "-fPIE", "-pie", "-I", build.INCLUDE, str(src), *objs, "-o", str(exe),
                    "-Wl,--unresolved-symbols=ignore-all", "-pthread"], check=True)
    return str(exe)


@pytest.mark.parametrize("conv", ["", "mma"])
@pytest.mark.parametrize("how", ["one", "threads"])
def test_every_layer_launches_on_both_devices(program, conv, how):
    env = dict(os.environ, FIT_CONV=conv)
    r = subprocess.run([program, how], env=env, capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout + r.stderr
