"""The value-norm warps of the score kernel when a wait gives up in the middle of a chunk: a chunk whose rows
have not all been seen must not count as done, for other CTAs take a head's norm once all its chunks do.  The
warps' loop is compiled for the host from the kernel's source, one lane, with waits that fail on order."""
import os
import re
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CUDA = os.environ.get("CUDA_HOME", "/usr/local/cuda")

MAIN = """
#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstring>
#include <vector_types.h>
using std::min;
constexpr int kTile = 128, kVRows = 32, kVWarps = 2, kRing = 16, kFirstV = 25, warp = 25, lane = 0;
struct S { static constexpr int kV = 4, kBlocks = 2; static constexpr uint32_t kOffV = 0, kVBytes = 32 * 256; };
struct Chunk { int ord, rhead, half, tile1, n1, n; };
struct Misc { unsigned long long v_full[8], v_empty[8]; Chunk ring[kRing]; } misc, *m = &misc;
static unsigned bits[8];
static int counted[8], waits, fail_at;
struct { const float* vbar_in; int split; unsigned* status; unsigned* vbar_bits; int* vcount; } p = {0, 0, 0, bits, counted};
static uint8_t store[S::kV * S::kVBytes], *gen = store;
static unsigned long long* smem_u32(unsigned long long* x) { return x; }
static bool wait_for(unsigned long long*, uint32_t, Misc*, unsigned*) { return ++waits != fail_at; }
static bool chunk_ready(Misc*, int, unsigned*) { return true; }
static void mbar_arrive(unsigned long long*) {}
static void __syncwarp() {}
static bool __all_sync(unsigned, bool x) { return x; }
static float __shfl_xor_sync(unsigned, float x, int) { return x; }
static unsigned __float_as_uint(float x) { unsigned u; memcpy(&u, &x, 4); return u; }
static void atomicMax(unsigned* a, unsigned x) { *a = std::max(*a, x); }
static void red_add_release(int* a, int x) { *a += x; }
static void give_up(Misc*, unsigned*) {}
static void mma_bf16_16816(float&, float&, float&, float&, unsigned, unsigned, unsigned, unsigned, unsigned, unsigned) {}
int main() {
  const int nchunks = 3, pieces = 8;  // chunks of two tiles, four pieces a tile
  for (int j = 0; j < nchunks; ++j) misc.ring[j] = {j, j, 0, 2 * j, 2, 3 * 256};
  for (fail_at = 1; fail_at <= nchunks * pieces + 1; ++fail_at) {
    waits = 0;
    memset(counted, 0, sizeof counted);
    [&] {
%s
    }();
    const int done = (fail_at - 1) / pieces;  // chunks whose waits have all ended
    for (int j = 0; j < nchunks; ++j)
      if (counted[j] != (j < done ? 1 : 0)) { printf("wait %%d: chunk %%d\\n", fail_at, j); return 1; }
  }
  puts("only whole chunks");
}
"""


@pytest.mark.skipif(shutil.which("g++") is None, reason="needs a host compiler")
def test_a_chunk_that_was_given_up_does_not_count(tmp_path):
    src = open(os.path.join(ROOT, "paper_2509_09754_b200", "csrc", "score_sm100.cu")).read()
    loop = re.search(r"    if \(!p\.vbar_in\) \{\n      const int vw = .*?\n    \}\n", src, re.S).group(0)
    cpp = tmp_path / "norms.cpp"
    cpp.write_text(MAIN % loop)
    exe = str(tmp_path / "norms")
    subprocess.run(["g++", "-std=c++17", "-O1", "-w", "-I", os.path.join(CUDA, "include"), str(cpp), "-o", exe], check=True)
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0 and r.stdout.strip() == "only whole chunks", r.stdout
