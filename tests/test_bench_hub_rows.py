"""bench.py's own binning of rows against the library's, hub rows included (no
GPU): which rows of many entries the numeric pass moves to its largest CTA
kernel depends on how many of them a product has."""
from __future__ import annotations

import os
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include <cstdio>
#include <vector>
#include "internal.h"
using namespace hs;
// stdin: "f c entries" per row; stdout: the hub constants, then each row's numeric key, the hub rows moved
int main() {
  const BinCfg b = numeric_bins(product_bins(bin_config(4), 1 << 20, 4), 1 << 20);
  std::vector<int> key;
  std::vector<long long> entries;
  long long f, c, e;
  int rows[HUB_LEVELS] = {0};
  while (scanf("%lld %lld %lld", &f, &c, &e) == 3) {
    key.push_back(row_key(f, c, e, b));
    entries.push_back(e);
    const int l = hub_level(key.back(), e);
    if (l >= 0) ++rows[l];
  }
  printf("%lld %d %d %d\n", (long long)HUB_ENTRIES, HUB_LEVELS, HUB_ROWS, KEY_LARGE);
  for (size_t i = 0; i < key.size(); ++i) printf("%d\n", hub_key(key[i], entries[i], hub_from(rows)));
  return 0;
}
"""


@pytest.mark.parametrize("hubs", [[], [(5000, 40)], [(5000, 300), (20000, 5)], [(5000, 300), (20000, 4)], [(70000, 400)]])
def test_bench_moves_the_rows_that_the_library_moves(tmp_path, hubs):
    import bench
    from paper_1109_3739_gb300 import build
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    lib = build.build()
    src, exe = tmp_path / "hubs.cu", tmp_path / "hubs"
    src.write_text(PROGRAM)
    libdir = os.path.dirname(lib)
    r = subprocess.run([nvcc, "-std=c++17", "-O1", "-I", os.path.join(ROOT, "paper_1109_3739_gb300", "csrc"), "-I",
                        os.path.join(ROOT, "include"), str(src), "-o", str(exe), "-L", libdir, "-lhspgemm", "-Xlinker",
                        f"-rpath={libdir}"], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-2000:]
    rng = np.random.default_rng(5)
    rows = [(f, max(1, f // d), min(f, e)) for f in (1, 32, 100, 600, 3000, 9000, 50000) for d in (1, 3, 50)
            for e in (1, 4096, 4097, 30000)]
    rows += [(int(n * 1.5), int(rng.integers(1, 2000)), n) for n, count in hubs for _ in range(count)]
    f, c, e = (np.array(x, dtype=np.int64) for x in zip(*rows))
    out = subprocess.run([str(exe)], input="".join(f"{a} {b} {d}\n" for a, b, d in rows), capture_output=True, text=True,
                         timeout=60)
    assert out.returncode == 0, out.stderr
    lines = out.stdout.split()
    assert [int(x) for x in lines[:3]] == [bench.HUB_ENTRIES, bench.HUB_LEVELS, bench.HUB_ROWS]
    keys = np.array([int(x) for x in lines[4:]])
    t = dict(warp_s_max=128, mid_s_max=1024, large_s_max=4096, sym_mid_s_max=1024, sym_heavy_from=0, sort_max=1024,
             sort_pct=50, num_heavy_from=0)
    got = bench.bin_rows(t, f, c, entries=e)
    assert (got["numeric_large"] == (keys == int(lines[3]))).all()
    count = sum(v.astype(int) for k, v in got.items() if k.startswith("numeric_"))
    assert (count == 1).all()
    assert (bench.bin_rows(t, f, c, entries=np.ones_like(e))["numeric_large"] == bench.bin_rows(t, f, c)["numeric_large"]).all()
