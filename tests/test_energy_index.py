"""The energy kernels' row numbers over element ranges up to the largest count a mesh may
have (2^31 - 1 tetrahedra), by a host program on the kernels' own index function."""
from __future__ import annotations

import os
import subprocess

from paper_0901_1024_gb300 import build as b

PROGRAM = r"""
#include <cstdio>
#include <cstdint>
#include "device.h"
using namespace dgdev;
int main() {
  long long k0, k1;
  while (std::scanf("%lld %lld", &k0, &k1) == 2) {
    const __int128 rows = __int128(6) * (k1 - k0);
    if (energy_rows(int(k0), int(k1)) != rows) { std::printf("rows of %lld %lld\n", k0, k1); return 1; }
    // 8 blocks an SM, 256 rows each: one step past the end fits the index chosen
    const long long step = 8LL * 152 * 256;
    const bool i32 = energy_index32(energy_rows(int(k0), int(k1)), step);
    if (i32 && __int128(unsigned(rows + step)) != rows + step) { std::printf("steps of %lld %lld\n", k0, k1); return 1; }
    if (!i32 && rows < 4000000000LL) { std::printf("64 bits for %lld %lld\n", k0, k1); return 1; }
    for (int c = 0; c < 6; ++c)
      for (long long k : {0LL, 1LL, (k1 - k0) / 2, k1 - k0 - 1}) {
        if (k >= k1 - k0) continue;
        const int64_t g = int64_t(c) * (k1 - k0) + k;
        const EnergyRow r = i32 ? energy_row<unsigned>(unsigned(g), int(k0), int(k1))
                                : energy_row<int64_t>(g, int(k0), int(k1));
        if (r.c != c || r.k != k) { std::printf("row %d %lld of %lld %lld\n", c, k, k0, k1); return 1; }
      }
  }
  return 0;
}
"""

# one and a few elements; around 2^32 / 6, where 32-bit row numbers end; the largest mesh
RANGES = [(0, 1), (3, 5), (10, 23), (0, 82944), (0, 715827881), (0, 715827882), (0, 715827883),
          (1, 715827990), (5, 2**31 - 1), (0, 2**31 - 1)]


def test_rows_of_every_range(tmp_path):
    src, exe = os.path.join(tmp_path, "i.cu"), os.path.join(tmp_path, "i")
    with open(src, "w") as f:
        f.write(PROGRAM)
    subprocess.run([b._nvcc(), *b.ARCH, *b.FLAGS, src, "-o", exe], check=True, capture_output=True)
    p = subprocess.run([exe], input="\n".join(f"{a} {z}" for a, z in RANGES), text=True,
                       capture_output=True)
    assert p.returncode == 0, p.stdout
