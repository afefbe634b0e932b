"""The scratch's bookkeeping when a device allocation fails, on the host with an allocator that
has a limit: a capacity above zero always has its arrays, and a smaller batch runs afterwards."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2206_11535_gb300", "csrc")
CUDA = os.path.join(os.path.dirname(os.path.dirname(os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc"))), "include")

PROGRAM = r"""
#include <cstdio>
#include <map>
#include "m3e_scratch.h"
using namespace m3e;

static std::map<char*, size_t> blocks;  // allocations and their sizes; nothing is touched
static size_t used = 0, limit = 0, next_at = 4096;
static int calls = 0, fail_at = -1;      // the call that fails, counted from 0
static int get(void** p, size_t bytes) {
  const bool no = calls++ == fail_at || used + bytes > limit;
  *p = no ? nullptr : (void*)next_at;
  if (no) return M3E_ENOMEM;
  blocks[(char*)next_at] = bytes;
  next_at += bytes + 4096;
  used += bytes;
  return M3E_OK;
}
static int put(void* p) {
  if (!p) return M3E_OK;
  auto it = blocks.find((char*)p);
  if (it == blocks.end()) { printf("released twice\n"); return M3E_ECUDA; }
  used -= it->second;
  blocks.erase(it);
  return M3E_OK;
}
static const ScratchMemory M = {get, put};

static size_t room(const void* p) { auto it = blocks.find((char*)p); return it == blocks.end() ? 0 : it->second; }
// every capacity is backed by its arrays, and the capacities are those of a batch of nf frames when ok
static bool sound(const Scratch& s) {
  return room(s.defer) >= 4 * (size_t)s.defer_cap && room(s.defer2) >= 4 * (size_t)s.defer_cap &&
         room(s.defer1b) >= 4 * (size_t)s.defer_cap && room(s.hf) >= 16 * (size_t)s.hits_cap &&
         room(s.hidx) >= 2 * (size_t)s.hits_cap && room(s.l3) >= 2 * (NB + 2) * (size_t)s.frames_cap &&
         room(s.fint) >= 16 * (size_t)s.frames_cap && room(s.fcbase) >= 8 * (size_t)s.frames_cap &&
         room(s.trip) >= 16 * (size_t)s.trip_cap && room(s.tek) >= 8 * (size_t)s.trip_cap &&
         room(s.trec) >= 32 * (size_t)s.trip_cap && room(s.combo) >= 16 * (size_t)s.combo_cap;
}
static bool holds(const Scratch& s, int64_t nf) {
  return s.work && s.counters && s.defer_cap >= nf && s.frames_cap >= nf && s.hits_cap >= 128 * nf &&
         s.trip_cap >= 64 * nf && s.combo_cap >= 192 * nf;
}
#define CHECK(x) do { if (!(x)) { printf("line %d: %s\n", __LINE__, #x); return 1; } } while (0)
"""


def _run(tmp_path, body):
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(PROGRAM + "int main() {\n" + body + "\nreturn 0;\n}\n")
    subprocess.run(["g++", "-std=c++17", "-O1", "-I" + CSRC, "-I" + os.path.join(ROOT, "include"), "-I" + CUDA, str(src),
                    "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0 and r.stdout == "", r.stdout


@pytest.mark.parametrize("first", [0, 5000])
def test_every_failing_allocation_leaves_a_usable_scratch(tmp_path, first):
    """The k-th allocation of a growth fails, for every k: the arrays of the capacities are there,
    then a smaller batch and at last the large one get their scratch."""
    _run(tmp_path, r"""
for (int k = 0; k < 40; ++k) {
  Scratch s;
  limit = (size_t)1 << 62; fail_at = -1;
  if (FIRST) CHECK(ensure_scratch(M, s, FIRST, true) == M3E_OK);
  calls = 0; fail_at = k;
  const int rc = ensure_scratch(M, s, 70000, true);
  CHECK(sound(s));
  CHECK(rc == M3E_OK ? holds(s, 70000) : rc == M3E_ENOMEM);
  fail_at = -1;
  for (int64_t nf : {20000, 70000}) {
    CHECK(ensure_scratch(M, s, nf, true) == M3E_OK);
    CHECK(sound(s) && holds(s, nf));
  }
  free_scratch(M, s);
  CHECK(used == 0 && blocks.empty());
}""".replace("FIRST", str(first)))


@pytest.mark.parametrize("nf", [9000, 200_000, 700_000])
def test_a_batch_that_fits_with_the_first_figures_runs(tmp_path, nf):
    """Memory for the first figures per frame but not for the roomy ones: the batch gets the first,
    keeps them on the next call, and a smaller batch, or a larger limit, gets the roomy ones."""
    _run(tmp_path, r"""
Scratch s;
limit = (size_t)1 << 62;
CHECK(ensure_scratch(M, s, NF, true) == M3E_OK && sound(s) && s.hits_cap > 128 * NF && s.trip_cap > 64 * NF);
const size_t roomy = used;
free_scratch(M, s);
limit = roomy - 1;
CHECK(ensure_scratch(M, s, NF, true) == M3E_OK && sound(s) && holds(s, NF));
CHECK(s.hits_cap == 128 * NF && s.trip_cap == 64 * NF && s.combo_cap == 192 * NF);
const size_t lean = used;
const void* hf = s.hf;
calls = 0;
CHECK(ensure_scratch(M, s, NF, true) == M3E_OK && calls == 0 && s.hf == hf);
CHECK(ensure_scratch(M, s, NF / 2, true) == M3E_OK && calls == 0 && s.hf == hf);
free_scratch(M, s);
limit = lean - 1;  // not even the first figures
CHECK(ensure_scratch(M, s, NF, true) == M3E_ENOMEM && sound(s));
CHECK(ensure_scratch(M, s, NF / 8, true) == M3E_OK && sound(s) && holds(s, NF / 8) && s.hits_cap >= 384 * (NF / 8));
limit = 3 * roomy;
CHECK(ensure_scratch(M, s, NF, true) == M3E_OK && sound(s) && s.hits_cap > 128 * NF);
free_scratch(M, s);
CHECK(used == 0);""".replace("NF", str(nf)))
