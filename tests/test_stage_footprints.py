"""What the tensor-core stage kernels ask of an SM, from the headers by a host program:
no two CTAs that could share an SM may want more tensor memory than it has, since a CTA
signals the next kernel before it allocates (launch.cuh)."""
from __future__ import annotations

import itertools
import os
import subprocess

import pytest

from paper_0901_1024_gb300 import build as b

PROGRAM = r"""
#include <cstdio>
#include <vector>
#include "tc_stage.cuh"
#include "tc_stage_t.cuh"
using namespace dgdev;
template <class D> void form(const char* name, int columns) {
  std::printf("%s %d %d\n", name, columns, tc_smem(columns, D::SMEM));
}
int main() {
  form<TcDims<1>>("N1", TcDims<1>::TMEM);
  form<TcDims<2>>("N2", TcDims<2>::TMEM);
  form<TcDims<2, true>>("N2pair", TcDims<2, true>::TMEM);
  form<TcDims<3>>("N3", TcDims<3>::TMEM);
  form<TcDims<3, true>>("N3pair", TcDims<3, true>::TMEM);
  form<TcDims<4>>("N4", TcDims<4>::TMEM);
  form<TtDims<5>>("N5", 512);
  form<TtDims<6>>("N6", 512);
  form<TtDims<7>>("N7", 512);
  // shared memory of the launch of 1, 65, 152, 153 and 14 000 tiles on 152 SMs
  for (int tiles : {1, 65, 152, 153, 14000})
    std::printf("alone%d %d %d\n", tiles, tc_cta_alone(tiles, 152) ? 1 : 0,
                tc_cta_alone(tiles, 152) ? tc_smem(512, TcDims<2, true>::SMEM) : 0);
  for (int N = 1; N <= 4; ++N)
    for (int tiles : {1, 152, 153, 304, 360, 381, 400, 455, 456, 608, 680, 700, 759, 760, 1000, 7317})
      std::printf("pair%d_%d %d %d\n", N, tiles, tc_paired(N, tiles, 152, false) ? 1 : 0,
                  tc_paired(N, tiles, 152, true) ? 1 : 0);
  // rings of K elements whose neighbours lie `hop` elements on, boundary faces among them
  for (int K : {1000, 50000})
    for (int hop : {1, 21999, 22001, 24999}) {
      std::vector<int32_t> nbr(4 * K);
      std::vector<signed char> code(4 * K);
      for (int i = 0; i < 4 * K; ++i) {
        const int k = i / 4;
        nbr[i] = (k + (i % 4 < 2 ? hop % K : K - hop % K)) % K;
        code[i] = i % 4 == 3 ? -1 : 5;
      }
      std::printf("far%d_%d %d 0\n", K, hop, scattered_mesh(nbr.data(), code.data(), K) ? 1 : 0);
    }
}
"""

SM_SMEM, CTA_SMEM, SM_COLUMNS = 228 * 1024, 1024, 512


@pytest.fixture(scope="module")
def forms(tmp_path_factory):
    d = tmp_path_factory.mktemp("footprints")
    src, exe = os.path.join(d, "f.cu"), os.path.join(d, "f")
    with open(src, "w") as f:
        f.write(PROGRAM)
    subprocess.run([b._nvcc(), *b.ARCH, *b.FLAGS, src, "-o", exe], check=True, capture_output=True)
    out = subprocess.run([exe], check=True, capture_output=True, text=True).stdout
    return {n: (int(c), int(s)) for n, c, s in (line.split() for line in out.splitlines())}


def signals_first(source):
    """Whether a kernel of this source signals the next grid before it allocates."""
    text = open(os.path.join(b.CSRC, source)).read()
    signal, alloc = text.find("pdl_launch_dependents();"), text.find("tc::tmem_alloc(&s_tmem")
    return signal >= 0 and (alloc < 0 or signal < alloc or text.count("pdl_launch_dependents();") > 1)


def test_no_cta_waits_for_columns_that_its_successor_holds(forms):
    """CTAs that fit an SM together may want more columns than it has only if both have theirs
    before their grids let the next one start (orders 1 to 4; 5 to 7 signal first)."""
    assert not signals_first("tc_stage.cuh")
    assert not signals_first("mixed_tc.cu")
    for k in (2, 3):
        for group in itertools.combinations_with_replacement(
                [n for n in forms if n[0] == "N"], k):
            smem, columns = (sum(forms[n][i] for n in group) for i in (1, 0))
            if smem + k * CTA_SMEM <= SM_SMEM and columns > SM_COLUMNS:
                assert all(n[1] in "1234" for n in group), group
    for n in ("N2pair", "N3pair"):             # the paired forms fit twice, no more
        assert 2 * (forms[n][1] + CTA_SMEM) <= SM_SMEM < 3 * (forms[n][1] + CTA_SMEM)


def test_a_wave_or_less_has_one_cta_an_sm(forms):
    """Up to one tile an SM no SM may take two CTAs while another idles."""
    for tiles in (1, 65, 152):
        alone, smem = forms[f"alone{tiles}"]
        assert alone == 1 and 2 * (smem + CTA_SMEM) > SM_SMEM
    assert forms["alone153"][0] == 0 and forms["alone14000"][0] == 0


def test_which_launches_are_paired(forms):
    """On 152 SMs: order 2 always, order 3 where two CTAs an SM measured faster (no worse than
    1 % slower), orders 1 and 4 never."""
    for tiles in (1, 152, 153, 304, 360, 381, 400, 455, 456, 608, 680, 700, 759, 760, 1000, 7317):
        assert [forms[f"pair{N}_{tiles}"][0] for N in (1, 2, 4)] == [0, 1, 0]
        single = tiles <= 152 or 380 < tiles < 456 or 684 < tiles < 760
        assert forms[f"pair3_{tiles}"][0] == (0 if single else 1), tiles
        # a mesh whose neighbours are scattered: order 3 never
        assert [forms[f"pair{N}_{tiles}"][1] for N in (1, 2, 3, 4)] == [0, 1, 0, 0]


def test_which_meshes_are_scattered(forms):
    """Faces over 22 000 elements away count, of every (1 + K / 8 192)th element; rings wrap, so
    a hop h is h or K - h away."""
    for K in (1000, 50000):
        for hop in (1, 21999, 22001, 24999):
            h, interior, far = hop % K, 0, 0
            for k in range(0, K, 1 + K // 8192):
                for n in ((k + h) % K, (k + h) % K, (k + K - h) % K):
                    interior += 1
                    far += abs(n - k) > 22000
            assert forms[f"far{K}_{hop}"][0] == int(2 * far > interior), (K, hop)
