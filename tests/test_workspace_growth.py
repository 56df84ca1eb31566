"""The context's workspace on the CPU, with the runtime's allocation calls stood in for: a growth
that fails leaves no capacity that nothing stands behind, and a later, smaller call has its
workspace again; blocks that a captured call may have been given outlive their growth."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2007_00308_gb300", "csrc")
NVCC = os.environ.get("NVCC") or "/usr/local/cuda/bin/nvcc"

MAIN = r"""
#include <cstdio>
#include <cstdlib>
#include <map>
#include "ps_internal.cuh"

static std::map<char*, size_t> live;   // device blocks, host memory here
static size_t most = (size_t)-1;       // larger allocations fail
static int errors = 0, freed = 0;
static cudaError_t last = cudaSuccess;
static cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
extern "C" {
cudaError_t __wrap_cudaMalloc(void** p, size_t n) {
  if (n > most) return last = cudaErrorMemoryAllocation;
  *p = malloc(n);
  live[(char*)*p] = n;
  return cudaSuccess;
}
cudaError_t __wrap_cudaFree(void* p) {
  if (p && !live.erase((char*)p)) ++errors;  // unknown, or freed twice
  ++freed;
  free(p);
  return cudaSuccess;
}
cudaError_t __wrap_cudaGetDevice(int* d) { *d = 0; return cudaSuccess; }
cudaError_t __wrap_cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) { *v = 152; return cudaSuccess; }
cudaError_t __wrap_cudaMemset(void*, int, size_t) { return cudaSuccess; }
cudaError_t __wrap_cudaGetLastError() { cudaError_t e = last; last = cudaSuccess; return e; }
cudaError_t __wrap_cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus* s) {
  *s = capture;
  return cudaSuccess;
}
}

// n bytes at p lie in a live block
static bool backed(const void* p, size_t n) {
  auto it = live.upper_bound((char*)p);
  if (!p || it == live.begin()) return false;
  --it;
  return (char*)p + n <= it->first + it->second;
}
#define CHECK(x) do { if (!(x)) { printf("line %d: %s\n", __LINE__, #x); ++errors; } } while (0)
// every capacity that the context claims has memory behind it
static void consistent(ps_context* c) {
  CHECK(c->tile_cap == 0 || (backed(c->d_counters, 64) && backed(c->d_tile_state, sizeof(TileState) * c->tile_cap) &&
                             (char*)c->d_tile_state == (char*)c->d_counters + 64));
  CHECK(c->rec_cap == 0 || backed(c->d_recs, (sizeof(LinkRec) + 4) * c->rec_cap));
  CHECK(c->pair_cap == 0 || backed(c->d_bin, 4 * c->pair_cap));
  CHECK(c->quad_hits_cap == 0 || backed(c->d_quad_hits, 8 * c->quad_hits_cap));
  const int64_t t = c->raster_tile_cap;
  CHECK(t == 0 || (backed(c->d_tile_count, 4 * (t + 1)) && backed(c->d_tile_off, 4 * (t + 1)) &&
                   backed(c->d_tile_cursor, 8 * (t + 1)) && backed(c->d_tile_list, 4 * (t + 1))));
}
"""

GROWTH = MAIN + r"""
int main() {
  ps_context* c = nullptr;
  CHECK(ps_create(&c) == PS_OK);
  consistent(c);
  const int64_t small = 1000, big = 50000000;
  for (int kind = 0; kind < 4; ++kind) {
    auto reserve = [&](int64_t n) {
      return ps_reserve(c, kind == 0 ? n : 0, kind == 1 ? n : 0, kind == 2 ? n : 0, kind == 3 ? n : 0);
    };
    // (what a failing growth of several blocks has done by then differs with the limit)
    for (size_t limit : {1000000ul, 100000000ul, 300000000ul, 500000000ul}) {
      most = (size_t)-1;
      CHECK(reserve(small) == PS_OK);
      consistent(c);
      most = limit;
      reserve(big);
      consistent(c);
      CHECK(reserve(small) == PS_OK);
      CHECK(cudaGetLastError() == cudaSuccess);  // or the next launch reports it as its own
      consistent(c);
      CHECK(c->tile_cap > 0);  // the counters are every call's
    }
  }
  ps_destroy(c);
  CHECK(live.empty());
  return errors ? 1 : 0;
}
"""


TESSELLATE_ONLY = MAIN + r"""
int main() {
  ps_context* c = nullptr;
  CHECK(ps_create(&c) == PS_OK);
  most = 100000000;  // the tile states of 50 M ribs, but not 9 bytes for each
  CHECK(ps_reserve(c, 1000, 50000000, 1000, 1000) == PS_OK);
  consistent(c);
  CHECK(c->tile_cap > 50000000 / 512 && c->pair_cap >= 1000 && c->rec_cap >= 1000 && c->quad_hits_cap == 0);
  CHECK(ps_reserve(c, 0, 5000000, 0, 0) == PS_OK);
  consistent(c);
  CHECK(c->quad_hits_cap >= 5000000);
  ps_destroy(c);
  return errors ? 1 : 0;
}
"""

CAPTURED = MAIN + r"""
int main() {
  ps_context* c = nullptr;
  CHECK(ps_create(&c) == PS_OK);
  auto reserve = [&](int64_t n) { return ps_reserve(c, n, n, n, n); };
  auto blocks = [&](void** b) {
    void* all[] = {c->d_counters, c->d_recs, c->d_bin, c->d_quad_hits, c->d_tile_count, c->d_tile_off,
                   c->d_tile_cursor, c->d_tile_list};
    for (int i = 0; i < 8; ++i) b[i] = all[i];
  };
  void *before[8], *after[8];
  ps_on_stream(c, nullptr);
  CHECK(reserve(2000) == PS_OK);
  const size_t count = live.size();
  CHECK(reserve(100000) == PS_OK);  // no capture yet: the blocks go
  CHECK(live.size() == count);
  blocks(before);
  capture = cudaStreamCaptureStatusActive;
  ps_on_stream(c, nullptr);
  capture = cudaStreamCaptureStatusNone;
  ps_on_stream(c, nullptr);
  size_t sum = 0;
  for (int64_t n = 100000; n < 4000000; n += 5000) {  // many small steps
    CHECK(reserve(n) == PS_OK);
    consistent(c);
  }
  blocks(after);
  for (int i = 0; i < 8; ++i) CHECK(after[i] != before[i] && backed(before[i], 1) && backed(after[i], 1));
  for (auto& b : live) sum += b.second;
  const size_t now = 64 + sizeof(TileState) * c->tile_cap + (sizeof(LinkRec) + 4) * c->rec_cap +
                     4 * c->pair_cap + 8 * c->quad_hits_cap + 20 * (c->raster_tile_cap + 1);
  CHECK(sum < 3 * now + 4096);
  ps_destroy(c);
  CHECK(live.empty());
  return errors ? 1 : 0;
}
"""


def run(tmp_path, source):
    src, exe = tmp_path / "main.cu", tmp_path / "main"
    src.write_text(source)
    wrap = []
    for name in ("Malloc", "Free", "GetDevice", "DeviceGetAttribute", "Memset", "GetLastError",
                 "StreamIsCapturing"):
        wrap += ["-Xlinker", f"--wrap=cuda{name}"]
    subprocess.run([NVCC, "-gencode", "arch=compute_103a,code=sm_103a", "-std=c++17", f"-I{CSRC}",
                    *wrap, "-o", str(exe), str(src), os.path.join(CSRC, "ps_api.cu")], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr


@pytest.fixture(autouse=True)
def _nvcc():
    if not os.path.exists(NVCC):
        pytest.skip("no nvcc")


def test_failed_growth_leaves_nothing_claimed(tmp_path):
    run(tmp_path, GROWTH)


def test_captured_blocks_are_kept(tmp_path):
    run(tmp_path, CAPTURED)


def test_reservation_without_room_for_the_words(tmp_path):
    run(tmp_path, TESSELLATE_ONLY)
