"""The buffers of a context on the host, with counted backing allocations: a
large piece of a slab that was given back serves the next request of its size,
giving back allocates no host memory, and pieces in use never overlap."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2510_12196_gb300", "csrc")

SOURCE = r"""
#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <map>
#include <new>

#include "devmem.h"

static long g_host = 0, g_obtained = 0, g_freed = 0;
void* operator new(size_t n) {
  g_host++;
  void* p = std::malloc(n);
  if (!p) throw std::bad_alloc();
  return p;
}
void operator delete(void* p) noexcept { std::free(p); }
void operator delete(void* p, size_t) noexcept { std::free(p); }

static char* g_next = reinterpret_cast<char*>(1 << 20);  // addresses only: nothing is accessed
void* gm::DevMem::obtain(size_t bytes) {
  g_obtained++;
  void* p = g_next;
  g_next += bytes + 4096;
  return p;
}
void gm::DevMem::raw_free(void*, size_t) noexcept { g_freed++; }

#define CHECK(x) \
  if (!(x)) return printf("%s\n", #x), 1

// a buffer of 300 KB from the end of the first slab, given back and wanted again
static int kept_piece() {
  gm::DevMem m;
  m.reserve(1 << 20);
  void* a = m.get(600 << 10);
  void* big = m.get(300 << 10);
  void* b = m.get(100 << 10);  // little of the slab is left
  m.put(big);
  const long before = g_obtained;
  CHECK(m.get(300 << 10) == big);
  CHECK(g_obtained == before);
  (void)a;
  (void)b;
  return 0;
}

// ten buffers of one size, then ten of another, all given back
static int quiet_put() {
  gm::DevMem m;
  m.reserve(4 << 20);
  for (size_t bytes : {(size_t)1000, (size_t)40000, (size_t)9000, (size_t)200000}) {
    void* p[10];
    for (auto& x : p) x = m.get(bytes);
    const long before = g_host;
    for (auto& x : p) m.put(x);
    CHECK(g_host == before);
  }
  m.release_all();
  return 0;
}

// random traffic: pieces in use are disjoint, everything obtained is freed
static int traffic(unsigned seed) {
  const long obtained = g_obtained, freed = g_freed;
  gm::DevMem m;
  m.reserve(3 << 20);
  std::map<char*, size_t> live;
  srand(seed);
  for (int i = 0; i < 4000; i++) {
    if (live.size() < 40 && rand() % 5 < 3) {
      const size_t bytes = (size_t)1 << (rand() % 20);
      const size_t want = bytes + (size_t)(rand() % 300);
      char* p = static_cast<char*>(m.get(want));
      CHECK(((uintptr_t)p & 255) == 0);
      auto hi = live.lower_bound(p);
      CHECK(hi == live.end() || p + want <= hi->first);
      if (hi != live.begin()) {
        --hi;
        CHECK(hi->first + hi->second <= p);
      }
      live[p] = want;
    } else if (!live.empty()) {
      auto it = live.begin();
      std::advance(it, rand() % live.size());
      m.put(it->first);
      live.erase(it);
    }
  }
  m.release_all();
  CHECK(g_obtained - obtained == g_freed - freed);
  CHECK(m.total == 0);
  return 0;
}

int main(int argc, char** argv) {
  if (argc > 1 && !strcmp(argv[1], "kept_piece")) return kept_piece();
  if (argc > 1 && !strcmp(argv[1], "quiet_put")) return quiet_put();
  for (unsigned s = 1; s <= 20; s++)
    if (traffic(s)) return 1;
  return 0;
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    cxx, cuda = shutil.which("g++"), "/usr/local/cuda/include"
    if not cxx or not os.path.exists(os.path.join(cuda, "cuda_runtime_api.h")):
        pytest.skip("no host compiler or CUDA headers")
    d = tmp_path_factory.mktemp("devmem")
    src, exe = d / "devmem.cpp", d / "devmem"
    src.write_text(SOURCE)
    # (256-byte alignment of the addresses above: slabs and allocations are multiples of 256)
    subprocess.run([cxx, "-O1", "-std=c++17", "-I", CSRC, "-I", cuda, str(src), "-o", str(exe)], check=True)
    return str(exe)


@pytest.mark.parametrize("what", ["kept_piece", "quiet_put", "traffic"])
def test_buffers(program, what):
    r = subprocess.run([program, what], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout
