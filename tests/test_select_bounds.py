"""Which memory the selection reads: its loads of keys, compiled for the host from the kernel's source with an
address checker, over every alignment of the array and every remainder of its length.  A vector load that
reaches past either end of the array ends the program."""
import os
import re
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CUDA = os.environ.get("CUDA_HOME", "/usr/local/cuda")

MAIN = """
#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <vector_types.h>
static void part(const unsigned* keys, int n) {
  %s
  for (int v = 0; v < n_vec; ++v) {
    const uint4 q = fetch(v);
    const unsigned x[4] = {q.x, q.y, q.z, q.w};
    for (int j = 0; j < 4; ++j) {
      const int e = 4 * v - mis + j;
      if (x[j] != (e >= 0 && e < n ? 1000u + e : 0u)) exit(2);
    }
  }
  if (n > 4 * n_vec - mis || 4 * n_vec - mis >= n + 4) exit(3);
}
int main() {
  for (int shift = 0; shift < 4; ++shift)
    for (int n = 1; n <= 37; ++n) {
      // the array starts `shift` elements behind a multiple of 16 bytes: what lies around it is not its own
      const int words = (n + shift + 3) / 4 * 4 + 4;
      unsigned* block = static_cast<unsigned*>(aligned_alloc(16, 4 * words));
      unsigned* keys = block + shift;
      for (int e = 0; e < n; ++e) keys[e] = 1000u + e;
      ASAN_POISON_MEMORY_REGION(block, shift * 4);
      ASAN_POISON_MEMORY_REGION(keys + n, (words - shift - n) * 4);
      part(keys, n);
      ASAN_UNPOISON_MEMORY_REGION(block, words * 4);
      free(block);
    }
  puts("inside");
}
"""


@pytest.mark.skipif(shutil.which("g++") is None, reason="needs a host compiler")
def test_key_loads_stay_inside_the_array(tmp_path):
    src = open(os.path.join(ROOT, "paper_2509_09754_b200", "csrc", "select.cu")).read()
    loads = re.search(r"  const int mis = .*?\n  auto fetch = .*?\n  };\n", src, re.S).group(0)
    cpp = tmp_path / "loads.cpp"
    cpp.write_text("#include <sanitizer/asan_interface.h>\n" + MAIN % loads)
    exe = str(tmp_path / "loads")
    subprocess.run(["g++", "-std=c++17", "-O1", "-g", "-fsanitize=address", "-I", os.path.join(CUDA, "include"),
                    str(cpp), "-o", exe], check=True)
    r = subprocess.run([exe], capture_output=True, text=True, env=dict(os.environ, ASAN_OPTIONS="detect_leaks=0"))
    assert r.returncode == 0 and r.stdout.strip() == "inside", r.stderr[:600]
