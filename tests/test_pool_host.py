"""The block pool's rules on the host, against a stand-in for the CUDA calls it
makes: a block is handed on only after its own device's work has completed,
whatever device is current, and what the pool keeps is bounded."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2504_10783_gb300", "csrc")

FAKE = r"""
#pragma once
#include <cstdlib>
#include <set>
#include <vector>
enum cudaError_t { cudaSuccess = 0, cudaErrorMemoryAllocation = 2, cudaErrorStreamCaptureUnsupported = 900 };
enum cudaStreamCaptureMode { cudaStreamCaptureModeGlobal, cudaStreamCaptureModeThreadLocal, cudaStreamCaptureModeRelaxed };
inline int g_dev = 0, g_sync_fails = 0;
inline cudaStreamCaptureMode g_mode = cudaStreamCaptureModeGlobal;
inline std::vector<int> g_synced;
inline std::set<void*> g_live, g_freed;
inline cudaError_t cudaGetDevice(int* d) { *d = g_dev; return cudaSuccess; }
inline cudaError_t cudaSetDevice(int d) { g_dev = d; return cudaSuccess; }
inline cudaError_t cudaGetLastError() { return cudaSuccess; }
inline cudaError_t cudaDeviceSynchronize() {
  g_synced.push_back(g_dev);
  return g_sync_fails ? cudaErrorStreamCaptureUnsupported : cudaSuccess;
}
inline cudaError_t cudaThreadExchangeStreamCaptureMode(cudaStreamCaptureMode* m) {
  const cudaStreamCaptureMode was = g_mode;
  g_mode = *m;
  *m = was;
  return cudaSuccess;
}
inline cudaError_t cudaMalloc(void** p, size_t) {
  *p = std::malloc(1);
  g_live.insert(*p);
  return cudaSuccess;
}
inline cudaError_t cudaFree(void* p) {
  g_live.erase(p);
  g_freed.insert(p);
  return cudaSuccess;
}
inline cudaError_t cudaMallocHost(void** p, size_t n) { return cudaMalloc(p, n); }
inline cudaError_t cudaFreeHost(void* p) { return cudaFree(p); }
"""

MAIN = r"""
#include <cstdio>
#include "ezo_pool.cuh"
#define EXPECT(c) do { if (!(c)) { std::printf("line %d: %s\n", __LINE__, #c); return 1; } } while (0)
using namespace ezo;
int main() {
  cudaError_t e;
  BlockPool pool(false);
  // completed work: the block is handed on, to one taker at a time
  void* a = pool.take(1000, &e);
  pool.give(a, true);
  EXPECT(pool.take(1000, &e) == a && pool.take(1000, &e) != a);
  // work that may still run: freed, not handed on
  pool.give(a, false);
  EXPECT(g_freed.count(a) && !g_live.count(a));
  // a block belongs to the device it was made on
  g_dev = 1;
  void* b = pool.take(1000, &e);
  pool.give(b, true);
  g_dev = 0;
  EXPECT(pool.take(1000, &e) != b);
  g_dev = 1;
  EXPECT(pool.take(1000, &e) == b);
  // the wait is for the given device; the current one is put back
  g_dev = 0;
  g_synced.clear();
  EXPECT(device_idle(1) && g_synced == std::vector<int>{1} && g_dev == 0);
  g_sync_fails = 1;
  EXPECT(!device_idle(1) && g_dev == 0 && !device_idle(0) && g_mode == cudaStreamCaptureModeGlobal);
  g_sync_fails = 0;
  // bounded: blocks kept, bytes kept, the largest block
  std::vector<void*> many;
  for (int i = 0; i < 40; ++i) many.push_back(pool.take(1000, &e));
  g_freed.clear();
  for (void* p : many) pool.give(p, true);
  EXPECT(g_freed.size() == 32);
  pool.trim();
  many.clear();
  for (int i = 0; i < 4; ++i) many.push_back(pool.take(32u << 20, &e));
  void* large = pool.take((32u << 20) + 1, &e);
  g_freed.clear();
  for (void* p : many) pool.give(p, true);
  pool.give(large, true);
  EXPECT(g_freed.size() == 3 && g_freed.count(large));
  pool.give(nullptr, true);
  // many small blocks do not keep a later one out: the longest unused go
  pool.trim();
  many.clear();
  for (int i = 0; i < 12; ++i) many.push_back(pool.take(1000, &e));
  for (void* p : many) pool.give(p, true);
  void* c = pool.take(8u << 20, &e);
  pool.give(c, true);
  EXPECT(!g_freed.count(c) && pool.take(8u << 20, &e) == c);
  return 0;
}
"""


@pytest.mark.skipif(shutil.which("g++") is None, reason="needs g++")
def test_pool_hands_on_only_idle_blocks(tmp_path):
    (tmp_path / "cuda_runtime.h").write_text(FAKE)
    (tmp_path / "main.cpp").write_text(MAIN)
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", str(tmp_path), "-I", CSRC, str(tmp_path / "main.cpp"), "-o",
                    str(tmp_path / "main"), "-lpthread"], check=True)
    r = subprocess.run([str(tmp_path / "main")], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
