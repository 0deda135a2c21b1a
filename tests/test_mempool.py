"""The pools of the set-up calls (csrc/mempool.cuh) against a device of limited memory, on the CPU: the
header is compiled with a stand-in for the CUDA runtime that counts its blocks and refuses what does not fit."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1801_05648_gb300", "csrc")

RUNTIME = r"""
#pragma once
#include <cstddef>
enum cudaError_t { cudaSuccess = 0, cudaErrorInvalidValue = 1, cudaErrorMemoryAllocation = 2 };
cudaError_t cudaMalloc(void** p, size_t bytes);
template <class T> cudaError_t cudaMalloc(T** p, size_t bytes) { return cudaMalloc(reinterpret_cast<void**>(p), bytes); }
cudaError_t cudaFree(void* p);
cudaError_t cudaGetLastError();
const char* cudaGetErrorString(cudaError_t e);
"""

MAIN = r"""
#include "mempool.cuh"
#include <cstdint>
#include <cstdio>
#include <cstdlib>

namespace {
size_t capacity = 0, used = 0;
std::map<void*, size_t> blocks;
std::mutex device;
cudaError_t last = cudaSuccess;
uintptr_t next_address = 1 << 20;
}  // namespace
cudaError_t cudaMalloc(void** p, size_t bytes) {
  std::lock_guard<std::mutex> g(device);
  if (used + bytes > capacity) return last = cudaErrorMemoryAllocation;
  *p = reinterpret_cast<void*>(next_address);
  next_address += bytes + 256;
  used += bytes;
  blocks[*p] = bytes;
  return cudaSuccess;
}
cudaError_t cudaFree(void* p) {
  std::lock_guard<std::mutex> g(device);
  if (!p) return cudaSuccess;
  auto it = blocks.find(p);
  if (it == blocks.end()) { std::printf("freed twice\n"); std::exit(1); }
  used -= it->second;
  blocks.erase(it);
  return cudaSuccess;
}
cudaError_t cudaGetLastError() { const cudaError_t e = last; last = cudaSuccess; return e; }
const char* cudaGetErrorString(cudaError_t) { return "error"; }

#define EXPECT(x) do { if (!(x)) { std::printf("line %d: %s (used %zu)\n", __LINE__, #x, used); std::exit(1); } } while (0)
using namespace fsi;
constexpr size_t MB = (size_t)1 << 20;

void give_up() {
  // what one context's pool holds is given up for another's allocation, or for one outside any pool
  capacity = 200 * MB;
  auto slabs = std::make_shared<Slabs>();
  auto a = std::make_shared<MemPool>(slabs), b = std::make_shared<MemPool>(std::make_shared<Slabs>());
  size_t got = 0, got2 = 0;
  void* p = a->take(120 * MB, got);
  a->give(p, got);
  EXPECT(used >= 120 * MB);
  void* again = a->take(118 * MB, got2);        // a released block serves a slightly smaller request
  EXPECT(again == p && got2 == got);
  a->give(again, got2);
  void* q = b->take(150 * MB, got2);
  EXPECT(used >= 150 * MB && used <= 180 * MB && cudaGetLastError() == cudaSuccess);
  b->give(q, got2);
  { DBuf<char> d(150 * MB); EXPECT(d.p); }
  // what cannot be had is an error with its code, and leaves none behind for the next launch's check
  bool thrown = false;
  try { a->take(300 * MB, got); } catch (const Error& e) { thrown = e.code == ENOMEM_; }
  EXPECT(thrown && cudaGetLastError() == cudaSuccess);
  thrown = false;
  DBuf<char> d;
  try { d.alloc(300 * MB); } catch (const Error& e) { thrown = e.code == ENOMEM_; }
  EXPECT(thrown && !d.p && d.n == 0 && cudaGetLastError() == cudaSuccess);
}

void bounds() {
  // a context's five pools together keep a limited amount, whichever of them it came from
  capacity = 100000 * MB;
  auto slabs = std::make_shared<Slabs>();
  std::vector<std::shared_ptr<MemPool>> pools;
  for (int i = 0; i < 5; ++i) pools.push_back(std::make_shared<MemPool>(slabs));
  for (int round = 0; round < 2; ++round) {
    std::vector<std::pair<void*, size_t>> b;
    for (auto& p : pools)
      for (int k = 0; k < 3; ++k) {
        size_t got = 0;
        void* x = p->take(200 * MB, got);
        b.emplace_back(x, got);
      }
    EXPECT(used >= 3000 * MB);
    for (size_t k = 0; k < b.size(); ++k) pools[k / 3]->give(b[k].first, b[k].second);
    for (auto& p : pools) p->settle();
    EXPECT(used > 0 && used <= 1024 * MB);
  }
  for (auto& p : pools) p->trim();
  EXPECT(used == 0);
  // small blocks: slabs up to a limit, then blocks of their own, all apart from each other and used again
  constexpr size_t kBlocks = 600, kBytes = 900 * 1024;
  for (int round = 0; round < 2; ++round) {
    std::map<uintptr_t, size_t> at;
    std::vector<std::pair<void*, size_t>> b;
    for (size_t k = 0; k < kBlocks; ++k) {
      size_t got = 0;
      void* x = pools[k % 5]->take(kBytes, got);
      EXPECT(got >= kBytes);
      auto next = at.lower_bound((uintptr_t)x);
      EXPECT(next == at.end() || (uintptr_t)x + kBytes <= next->first);
      EXPECT(next == at.begin() || std::prev(next)->first + kBytes <= (uintptr_t)x);
      at[(uintptr_t)x] = got;
      b.emplace_back(x, got);
    }
    EXPECT(used <= 8 * 32 * MB + kBlocks * 2 * MB);
    for (size_t k = 0; k < kBlocks; ++k) pools[k % 5]->give(b[k].first, b[k].second);
  }
  for (auto& p : pools) p->trim();
  EXPECT(used <= 8 * 32 * MB);
}

void slab_under_pressure() {
  // a slab that does not fit beside what its own context's pools hold
  capacity = 100 * MB;
  auto slabs = std::make_shared<Slabs>();
  MemPool a(slabs);
  size_t got = 0, small = 0;
  void* big = a.take(90 * MB, got);
  a.give(big, got);
  void* x = a.take(1024, small);
  EXPECT(x && small == 1024 && used == 32 * MB);
  a.give(x, small);
}

int main(int argc, char** argv) {
  const std::string what = argc > 1 ? argv[1] : "";
  if (what == "give_up") give_up();
  else if (what == "bounds") bounds();
  else if (what == "slab_under_pressure") slab_under_pressure();
  else return 2;
  EXPECT(used == 0 && blocks.empty());           // everything came back
  return 0;
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no g++")
    d = tmp_path_factory.mktemp("pool")
    (d / "cuda_runtime.h").write_text(RUNTIME)
    (d / "main.cpp").write_text(MAIN)
    exe = str(d / "pool")
    r = subprocess.run([cxx, "-std=c++20", "-g", "-pthread", "-I", str(d), "-I", CSRC, "-x", "c++", str(d / "main.cpp"),
                        "-o", exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-4000:]
    return exe


@pytest.mark.parametrize("what", ["give_up", "bounds", "slab_under_pressure"])
def test_pool(what, program):
    r = subprocess.run([program, what], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout + r.stderr
