"""Launch shapes of the FP64 x passes, asked of the rule itself (a host program built with nvcc, no GPU): at the
lengths with a compile-time schedule (blocks of 256 threads, two to an SM) no other number of rows per block has
fewer waves of blocks at no more rows for the busiest SM, or fewer rows at no more waves."""
import os
import subprocess

import pytest

from paper_1411_0330_gb300 import build

PROGRAM = r"""
#include <cstdio>
#include "internal.h"
using namespace lsh;
int main() {
  const int len[] = {16, 32, 48, 64, 96, 128, 256}, side[] = {1, 12, 16, 30, 32, 48, 64, 96, 128};
  for (int nx : len)
    for (int ny : side)
      for (int nz : side)
        for (int c : {2, 3, 6})
          for (int S : {1, 2, 3, 6, 12}) {
            if ((c == 2) != (nz == 1)) continue;
            Plan1D px, py, pz;
            if (!lsh_make_plan(nx, &px) || !lsh_make_plan(ny, &py) || !lsh_make_plan(nz, &pz)) return 1;
            const LaunchCfg L = pass_cfg<double>(nx, ny, nz, c, px, py, pz, S);
            std::printf("%d %d %d %d %d %d %d %d\n", nx, ny, nz, c, S, L.RY, L.thr_x, (int)L.smem_x);
          }
  return 0;
}
"""


@pytest.fixture(scope="module")
def shapes(tmp_path_factory):
    d = tmp_path_factory.mktemp("shapes")
    (d / "shapes.cu").write_text(PROGRAM)
    subprocess.run([build._nvcc(), *build.ARCH, "-std=c++17", "-O0", "-I" + build.CSRC,
                    "-I" + os.path.join(build.ROOT, "include"), "-o", str(d / "shapes"), str(d / "shapes.cu")],
                   check=True, capture_output=True)
    out = subprocess.run([str(d / "shapes")], check=True, capture_output=True, text=True).stdout
    return [tuple(int(v) for v in line.split()) for line in out.splitlines()]


def test_no_other_block_has_fewer_waves_and_no_more_rows(shapes):
    assert len(shapes) > 1000
    for nx, ny, nz, c, S, RY, threads, _ in shapes:
        rps, cap = c * ny * nz, max(2, 2 * (32768 // ((nx | 1) * 16)))
        if cap >= rps:
            continue  # a system is a block or two

        def cost(d):
            blocks = S * rps // d
            return -(-blocks // 304), -(-blocks // 152) * d

        assert rps % RY == 0 and RY <= cap and threads == 256
        got = cost(RY)
        for d in range(2, cap + 1, 2):
            if rps % d == 0:
                other = cost(d)
                assert not (other != got and other[0] <= got[0] and other[1] <= got[1]), (nx, ny, nz, c, S, RY, d)


def test_blocks_fit_in_shared_memory(shapes):
    for nx, ny, nz, c, S, RY, _, smem in shapes:
        assert smem + 13 * 1024 <= 113 * 1024, (nx, ny, nz, c, S, RY)  # two blocks to an SM
