"""The arena of a set-up at the end of the device's memory, on the CPU: its own
source with a cudaMalloc that hands out a fixed number of bytes."""

import os
import subprocess

import pytest

from paper_2406_19754_gb300 import build

# the three runtime calls the arena makes (2: cudaErrorMemoryAllocation); they
# take precedence over the shared runtime library's
DEVICE = r"""
#include <stdlib.h>
#include <map>

size_t room = 0;
static std::map<void*, size_t> held;
bool nothing_held() { return held.empty(); }

extern "C" int cudaMalloc(void** p, size_t bytes) {
  if (bytes > room) return 2;
  room -= bytes;
  held[*p = aligned_alloc(256, bytes)] = bytes;
  return 0;
}
extern "C" int cudaFree(void* p) {
  if (!held.count(p)) abort();
  room += held[p];
  held.erase(p);
  free(p);
  return 0;
}
extern "C" int cudaGetLastError() { return 0; }
"""

HARNESS = r"""
#include <stdio.h>
#include "common.cuh"

extern size_t room;
bool nothing_held();

#define WANT(c) do if (!(c)) { printf("line %d: %s\n", __LINE__, #c); return 1; } while (0)

int main() {
  const size_t M = 1 << 20, S = amg::ARENA_SLAB_MIN;
  amg::Arena ar;
  void *a, *b, *c;
  // a kept large block makes room for a slab
  room = 8 * M + S / 2;
  ar.begin_reuse();
  WANT(ar.alloc(&a, 8 * M) == AMG_OK);
  ar.release(a);
  WANT(ar.alloc(&b, 1000) == AMG_OK);
  WANT(room == 8 * M - S / 2);
  WANT(ar.alloc(&a, room) == AMG_OK && room == 0);
  WANT(ar.alloc(&c, 1000) == AMG_OK);  // from the same slab
  WANT(ar.alloc(&c, 3 * M) == AMG_ERR_OOM);
  ar.end_reuse();
  ar.release_all();
  WANT(room == 8 * M + S / 2 && nothing_held());
  // less room than a slab: a block of its own, kept and used again
  room = S / 2;
  ar.begin_reuse();
  WANT(ar.alloc(&a, S / 4) == AMG_OK && room == S / 4);
  WANT(ar.alloc(&b, S / 4) == AMG_OK && room == 0);
  WANT(ar.alloc(&c, 256) == AMG_ERR_OOM);
  ar.release(a);
  WANT(ar.alloc(&c, 256) == AMG_OK && room == S / 4 - 256);  // what was kept went back
  ar.end_reuse();
  ar.release_all();
  WANT(room == S / 2 && nothing_held());
  // a request larger than the first slab gets one that holds it
  room = 4 * M;
  ar.begin_reuse();
  WANT(ar.alloc(&a, M) == AMG_OK && room == 3 * M);
  ar.end_reuse();
  ar.release_all();
  WANT(room == 4 * M && nothing_held());
  return 0;
}
"""


def test_small_requests_when_memory_is_short(tmp_path):
    src, dev, exe = tmp_path / "arena.cu", tmp_path / "device.cpp", tmp_path / "arena"
    src.write_text(HARNESS)
    dev.write_text(DEVICE)
    try:
        nvcc = build.nvcc()
    except RuntimeError:
        pytest.skip("no nvcc")
    cmd = [nvcc, str(src), str(dev), os.path.join(build.CSRC, "util.cu"), "-o", str(exe)]
    cmd += build.ARCH + ["-std=c++17", "-I", build.INCLUDE, "-I", build.CSRC, "-cudart=shared",
                         "-Xlinker", "-rpath," + build._cuda_lib()]
    r = subprocess.run(cmd, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout + r.stderr
