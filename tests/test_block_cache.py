"""The host-side cache of scratch blocks (csrc/blocks.h), compiled for the CPU against a fake pool."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2206_00470_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include <map>
#include "blocks.h"
#define CHECK(c) do { if (!(c)) { std::printf("line %d: %s (kept %zu, allocs %d)\n", __LINE__, #c, cache.kept(), d.allocs); return 1; } } while (0)
struct Driver {            // blocks are numbers; `limit` bytes of device memory
  std::map<void*, size_t> live;
  size_t in_use = 0, limit = ~(size_t)0;
  int allocs = 0, frees = 0;
  char* next = (char*)4096;
};
struct Mem {
  Driver* d;
  int alloc(void** p, size_t n) {
    ++d->allocs;
    if (d->in_use + n > d->limit) return 2;
    *p = d->next; d->next += n; d->live[*p] = n; d->in_use += n;
    return 0;
  }
  void free(void* p) { if (!d->live.count(p)) std::abort(); ++d->frees; d->in_use -= d->live[p]; d->live.erase(p); }
};
int main() {
  const size_t M = 1u << 20;
  Driver d; Mem m{&d}; adapm::BlockCache cache; void *a, *b, *c;
  // reuse: the same size class again is no call into the pool
  CHECK(cache.take(m, 3000, false, &a) == 0 && d.allocs == 1);
  cache.give(m, a);
  CHECK(cache.take(m, 2900, false, &b) == 0 && b == a && d.allocs == 1 && cache.kept() == 0);
  cache.give(m, b);
  // large blocks and those of a graph are not kept
  CHECK(cache.take(m, 65 * M, false, &c) == 0); cache.give(m, c); CHECK(d.frees == 1);
  CHECK(cache.take(m, 3000, true, &c) == 0 && c != a); cache.give(m, c); CHECK(d.frees == 2);
  // full of sizes nobody asks for any more: the new size is kept all the same, the oldest goes
  void* p[32];
  for (int i = 0; i < 9; ++i) CHECK(cache.take(m, 60 * M, false, &p[i]) == 0);
  for (int i = 0; i < 9; ++i) cache.give(m, p[i]);
  CHECK(cache.kept() <= adapm::BlockCache::kKeep);
  for (int i = 0; i < 8; ++i) CHECK(cache.take(m, 40 * M, false, &p[i]) == 0);
  for (int i = 0; i < 8; ++i) cache.give(m, p[i]);
  int before = d.allocs;
  for (int i = 0; i < 8; ++i) CHECK(cache.take(m, 40 * M, false, &p[i]) == 0);
  CHECK(d.allocs == before);
  for (int i = 0; i < 8; ++i) cache.give(m, p[i]);
  CHECK(cache.kept() <= adapm::BlockCache::kKeep && d.in_use == cache.kept());
  // no memory: the kept blocks serve another size, small or large
  d.limit = d.in_use + M;
  CHECK(cache.take(m, 50 * M, false, &a) == 0 && cache.kept() == 0);
  cache.give(m, a);
  d.limit = 70 * M;
  CHECK(cache.take(m, 66 * M, false, &b) == 0 && cache.kept() == 0);
  // nothing kept: the error is the pool's
  CHECK(cache.take(m, 66 * M, false, &c) == 2);
  cache.give(m, b);
  CHECK(d.in_use == 0);
  CHECK(cache.take(m, 100, false, &a) == 0);
  cache.give(m, a);
  cache.release([&](void* q) { m.free(q); });
  CHECK(cache.kept() == 0 && d.in_use == 0 && d.live.empty());
  return 0;
}
"""


def test_blocks_are_reused_exchanged_and_given_back(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("g++ not available")
    src, exe = tmp_path / "blocks.cpp", tmp_path / "blocks"
    src.write_text(PROGRAM)
    r = subprocess.run([gxx, "-std=c++17", "-Wall", "-Werror", "-I", CSRC, str(src), "-o", str(exe)],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout
