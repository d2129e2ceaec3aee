"""Host check of the rules that choose a launch's route and size (no GPU): the
library's own functions, compiled for the host."""
from __future__ import annotations

import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def run(tmp_path, body):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    src, exe = tmp_path / "rule.cu", tmp_path / "rule"
    src.write_text('#include <cstdio>\n#include <set>\n#include "internal.h"\nusing namespace hs;\n'
                   "static int bad = 0;\n#define CHECK(x) do { if (!(x)) { ++bad; printf(\"line %d: %s\\n\", __LINE__, #x); } } while (0)\n"
                   "int main() {\n" + body + "\nreturn bad != 0;\n}\n")
    r = subprocess.run([nvcc, "-std=c++17", "-O1", "-I", os.path.join(ROOT, "paper_1109_3739_gb300", "csrc"), "-I",
                        os.path.join(ROOT, "include"), str(src), "-o", str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-2000:]
    out = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert out.returncode == 0, out.stdout


def test_spref_leaves_the_bitmap_where_b_is_wide(tmp_path):
    """Rows of B of more than 2048 entries cost the bitmap kernel a sweep for every 2^20 columns; without a bound
    a wide J made them several times slower than the radix sort."""
    run(tmp_path, r"""
  const int64_t tuples = 54000000, rows = 20000, entries = 50000000, M = 1 << 20;
  CHECK(!spref_by_radix(0, 0, tuples, 200000, 1LL << 31));      // no long row
  CHECK(!spref_by_radix(rows, entries, tuples, 200000, M));     // one sweep
  CHECK(spref_by_radix(rows, entries, tuples, 200000, 16 * M));
  CHECK(spref_by_radix(rows, entries, tuples, 200000, 32 * M));
  CHECK(!spref_by_radix(1, 3000, 4200000, 200000, 16 * M));     // one row beside millions of others' tuples
  CHECK(spref_by_radix(1, 200000, 4200000, 200000, 16 * M));
  CHECK(spref_by_radix(1, 3000, 3000, 1, (1LL << 31) - 1));     // two thousand sweeps for a few tuples
  CHECK(spref_by_radix(1 << 20, 2147483647LL, 2147483647LL, 1 << 20, (1LL << 31) - 1));
  for (int64_t n = 1; n < 1LL << 31; n = n * 3 / 2 + 1)           // wider never goes back to the bitmap
    for (int64_t r : {1, 151, 152, 153, 2000, 100000})
      for (int64_t len : {2049, 20000})
        CHECK(!spref_by_radix(r, r * len, 2 * r * len, 200000, n) ||
              spref_by_radix(r, r * len, 2 * r * len, 200000, n * 2));""")


def test_hub_rows_are_moved_while_they_are_few(tmp_path):
    """Rows of many entries of A take the kernel of 1024 threads, a block an SM, only as long as at most HUB_ROWS of
    them do: the longest ones where there are more."""
    run(tmp_path, r"""
  const int none[HUB_LEVELS] = {0}, few[HUB_LEVELS] = {3, 2, 1}, many[HUB_LEVELS] = {3000}, mixed[HUB_LEVELS] = {500, 100, 30, 5};
  const int edge[HUB_LEVELS] = {HUB_ROWS}, over[HUB_LEVELS] = {HUB_ROWS + 1}, all[HUB_LEVELS] = {9, 9, 9, 9, 9, 1000};
  CHECK(hub_from(none) == 0 && hub_from(few) == 0 && hub_from(edge) == 0);
  CHECK(hub_from(many) == 1 && hub_from(over) == 1);   // none of those: their level is 0
  CHECK(hub_from(mixed) == 1 && hub_from(all) == HUB_LEVELS);
  CHECK(hub_level(KEY_MID, HUB_ENTRIES) < 0 && hub_level(KEY_MID, HUB_ENTRIES + 1) == 0);
  CHECK(hub_level(KEY_MID, 4 * HUB_ENTRIES) == 0 && hub_level(KEY_MID, 4 * HUB_ENTRIES + 1) == 1);
  CHECK(hub_level(KEY_MID, 1LL << 40) == HUB_LEVELS - 1);
  for (int key : {0, KEY_TINY, KEY_LARGE, KEY_SPA, KEY_HEAVY, NKEYS - 1}) CHECK(hub_key(key, 1 << 20, 0) == key);
  BinCfg narrow{}, wide{};
  narrow.cap_large = 8192;
  wide.cap_large = 4096;
  CHECK(!hub_always(KEY_MID, narrow) && hub_always(KEY_MID, wide) && !hub_always(KEY_MID_S, wide) && hub_always(KEY_LARGE_S, narrow));
  for (int key = KEY_TINY + 1; key < KEY_SPA; ++key) {
    if (key == KEY_LARGE) continue;
    CHECK(hub_key(key, 5000, 0) == KEY_LARGE && hub_key(key, 5000, 1) == key && hub_key(key, 4096, 0) == key);
    CHECK(hub_key(key, 20000, 1) == KEY_LARGE && hub_key(key, 1LL << 40, HUB_LEVELS) == key);
  }""")


def test_symbolic_bitmap_sizes_are_few(tmp_path):
    """The launch sizes of the bitmap kernel hold B's columns and do not follow every width: each is asked of the
    runtime once and kept."""
    run(tmp_path, r"""
  std::set<int64_t> sizes;
  for (int64_t n = 1; n < 1LL << 31; n += n < 3000000 ? 1 : n / 7) {
    const int64_t w = sym_bitmap_words(n);
    CHECK(w * 32 >= (n < BITMAP_COLS ? n : BITMAP_COLS) && w <= BITMAP_COLS / 32);
    sizes.insert(w);
  }
  CHECK(sizes.size() <= 4);""")
