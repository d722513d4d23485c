"""Index words of the scattering renderer's traversal (csrc/gf_words.h, host code), on the CPU.

Every node index that a field below 2^26 primitives can have goes through a stack word and
back, none is taken for "no entry"; and the bound on the number of four-wide nodes holds on
radix trees that come near it.
"""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include <algorithm>
#include <cstdio>
#include <vector>
#include "gf_words.h"

// internal nodes at even depth of the radix tree over keys [a, b) (ties by position)
static int64_t even_nodes(const std::vector<uint64_t>& k, int64_t a, int64_t b, int depth) {
  if (b - a < 2) return 0;
  uint64_t x = k[a] ^ k[b - 1];
  int64_t m;
  if (x == 0) {  // equal keys: the tree of the positions
    uint64_t p = (uint64_t)a ^ (uint64_t)(b - 1);
    int h = 63 - __builtin_clzll(p);
    m = (int64_t)(((uint64_t)(b - 1) >> h) << h);
  } else {
    const int h = 63 - __builtin_clzll(x);
    const uint64_t first = (k[b - 1] >> h) << h;
    m = std::lower_bound(k.begin() + a, k.begin() + b, first) - k.begin();
  }
  return (depth % 2 == 0 ? 1 : 0) + even_nodes(k, a, m, depth + 1) + even_nodes(k, m, b, depth + 1);
}

static uint64_t spread(uint64_t v) {
  uint64_t r = 0;
  for (int i = 0; i < 10; ++i) r |= (v >> i & 1) << (3 * i);
  return r;
}

int main() {
  int bad = 0;
  const int64_t top = gf::max_nodes4(gf::kMaxPrims - 1) - 1;
  for (int64_t node : std::vector<int64_t>{0, 1, (1 << 26) - 1, 1 << 26, (1 << 26) + 12345, top})
    for (uint32_t slot = 0; slot < 32; ++slot) {
      const int held = (int)gf::index_word((uint32_t)node, slot);  // as the stack holds it
      const uint32_t w = (uint32_t)held;
      if (w == gf::kNoWord || (int64_t)gf::word_index(w) != node || gf::word_slot(w) != slot) {
        printf("node %lld slot %u: word %x\n", (long long)node, slot, w);
        ++bad;
      }
    }
  // regular grids of one class (a full tree of odd height is the worst), and equal keys
  for (int64_t nx : {1, 2, 8, 13, 20, 32, 64})
    for (int64_t ny : {1, 8, 21, 32, 64}) {
      const int64_t nz = nx == 64 && ny == 64 ? 8 : 32;
      std::vector<uint64_t> k;
      for (int64_t z = 0; z < nz; ++z)
        for (int64_t y = 0; y < ny; ++y)
          for (int64_t x = 0; x < nx; ++x)
            k.push_back(spread(x * 1024 / nx) << 2 | spread(y * 1024 / ny) << 1 | spread(z * 1024 / nz));
      std::sort(k.begin(), k.end());
      const int64_t n = (int64_t)k.size(), e = even_nodes(k, 0, n, 0);
      if (e > (2 * n - 1) / 3 || 2 * e + 72 > gf::max_nodes4(n)) { printf("grid %lld: %lld\n", (long long)n, (long long)e); ++bad; }
    }
  int64_t most = 0;
  for (int64_t n : {2, 3, 8, 32, 100, 8192, 100000}) {
    const std::vector<uint64_t> k(n, 7);
    const int64_t e = even_nodes(k, 0, n, 0);
    if (e > (2 * n - 1) / 3 || 2 * e + 72 > gf::max_nodes4(n)) { printf("equal keys %lld: %lld\n", (long long)n, (long long)e); ++bad; }
    most = std::max(most, 1000 * e / n);
  }
  if (most < 660) { printf("no tree near the bound: %lld\n", (long long)most); ++bad; }
  printf(bad ? "bad\n" : "ok\n");
  return bad != 0;
}
"""


def test_index_words(tmp_path):
    src = tmp_path / "words.cpp"
    src.write_text(PROGRAM)
    exe = tmp_path / "words"
    subprocess.run(["g++", "-std=c++17", "-O1", "-I",
                    os.path.join(ROOT, "paper_2602_05081_gb300", "csrc"), str(src), "-o", str(exe)],
                   check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0 and r.stdout.strip() == "ok", r.stdout
