"""Index arithmetic of the kernels, checked on the host: the same header
(csrc/cg_index.h) compiled as plain C++ against tables that refuse an index out
of range."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1604_06667_gb300", "csrc")

PRELUDE = r"""
#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <vector>
#include "cg_index.h"
#define CHECK(x) do { if (!(x)) { std::printf("line %d: %s\n", __LINE__, #x); std::exit(1); } } while (0)
template <class T>
struct Table {                       // an array that refuses an index out of range
  std::vector<T> v;
  explicit operator bool() const { return true; }
  const T& operator[](int64_t i) const {
    if (i < 0 || i >= (int64_t)v.size()) { std::printf("index %lld of %zu\n", (long long)i, v.size()); std::exit(1); }
    return v[(size_t)i];
  }
};
"""


def _run(tmp_path, body):
    cxx = shutil.which("g++") or pytest.skip("no host compiler")
    src, exe = str(tmp_path / "t.cpp"), str(tmp_path / "t")
    with open(src, "w") as f:
        f.write(PRELUDE + body)
    subprocess.run([cxx, "-std=c++17", "-O1", "-I", CSRC, src, "-o", exe], check=True)
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout


def test_shares_of_empty_slots(tmp_path):
    """Slots of a last 128-target tile whose second half is empty have no
    candidate count of their own."""
    _run(tmp_path, r"""
int main() {
  for (int P : {1, 63, 64, 65, 128, 129, 192, 193, 40000, 40001}) {
    const int slots = (P + 127) / 128 * 128;
    Table<uint32_t> perm;
    Table<int> cand;
    for (int s = 0; s < slots; ++s) perm.v.push_back(s < P ? (uint32_t)s : cg::kEmptySlot);
    for (int t = 0; t < (P + 63) / 64; ++t) cand.v.push_back(300 * (t % 5));
    for (int s = 0; s < slots; ++s) {
      const int n = cg::slot_shares(perm, cand, s, 64, 4);
      CHECK(n == (s < P ? cg::wide_shares(cand[s / 64], 4) : 0));
      CHECK(cg::slot_shares(perm, (const int*)nullptr, s, 64, 4) == (s < P ? 4 : 0));
    }
  }
}
""")


def test_kd_keys_fit_32_bits(tmp_path):
    """Up to 2^31 - 1 targets the node's number and the coordinate share 32 bits,
    the node above the coordinate."""
    _run(tmp_path, r"""
int main() {
  for (int64_t P : {(int64_t)4096, (int64_t)4097, ((int64_t)1 << 28) + 1, (int64_t)1 << 29, ((int64_t)1 << 29) + 1,
                    (int64_t)805306368, ((int64_t)1 << 30) + 1, ((int64_t)1 << 31) - 1}) {
    const int64_t tiles = (P + 127) / 128;
    const int top = cg::kd_top_levels(tiles, 128, 4096);
    CHECK(((tiles + ((int64_t)1 << top) - 1) >> top) * 128 <= 4096);
    for (int l = 0; l < top; ++l) {
      const int bits = cg::kd_coord_bits(l);
      CHECK(bits >= 8 && bits <= 16 && l + bits <= 32);
      const uint32_t last = (uint32_t)(((uint64_t)1 << l) - 1);      // the level's last node
      for (uint32_t node : {0u, last / 2, last}) {
        const uint64_t lo = cg::kd_key(node, l, 0.f), hi = cg::kd_key(node, l, 1.f);
        CHECK(lo == (uint64_t)node << bits && hi == lo + (1u << bits) - 1);
        CHECK(cg::kd_key(node, l, 0.25f) < cg::kd_key(node, l, 0.75f));
        CHECK((hi >> (l + bits)) == 0);
      }
    }
  }
}
""")


def test_folds_keep_chains_short(tmp_path):
    """Parts of a tile's candidates that are summed apart: at least two chunks, and
    no longer than n_fold equal ones, or than three chunks, whatever the total."""
    _run(tmp_path, r"""
int main() {
  for (int total : {0, 1, 63, 64, 65, 96, 97, 128, 200, 1000, 4097, 1 << 20, 2147483647})
    for (int n : {1, 2, 3, 29, 64}) {
      const int64_t k = cg::wide_fold_chunks(total, n, 32), chunks = ((int64_t)total + 31) / 32;
      CHECK(k >= 2);
      if (n == 1 || chunks < 4) CHECK(k >= chunks);
      else CHECK(k <= 3 || (k - 1) * n < chunks);
    }
}
""")
