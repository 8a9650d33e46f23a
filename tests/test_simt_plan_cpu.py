"""The work split of the float32 MTTKRP kernel (csrc/simt_plan.cuh), compiled for the
host: the tiles taken whole and the tiles cut into runs are the tiles of the output,
each once; the partial slots fit the scratch; and the tile height is the cheapest of
those planned one by one, whatever was tried before it.  Short outputs keep the GPU
busy with the scratch that a context sets aside."""
import math
import os
import random
import subprocess

import pytest

from _util import ROOT
from paper_1806_07985_gb300 import build

SOURCE = r"""
#include <cstdio>
#include "simt_plan.cuh"
using namespace nncp;
static void show(const SimtPlan& p) {
  printf(" %d %lld %lld %lld %d %d %d %lld %.17g", p.BM, p.a.whole, p.a.U2, p.a.nk, p.a.G2, p.a.two, p.grid,
         p.a.slot_floats, p.cost);
}
int main() {
  int N, R, lo, hi;
  long long cap, x;
  while (scanf("%d %d %d %d %lld", &N, &R, &lo, &hi, &cap) == 5) {
    KrpDesc KL = {}, KQ = {};
    int64_t L = 1, I = 1, Q = 1;
    for (int n = 0; n < N; ++n) {
      if (scanf("%lld", &x) != 1) return 1;
      if (n >= lo && n < hi) {
        I *= x;
        continue;
      }
      KrpDesc& d = n < lo ? KL : KQ;
      d.dim[d.nm++] = x;
      (n < lo ? L : Q) *= x;
    }
    SimtPlan p;
    if (plan_simt(L, I, Q, KL, KQ, R, cap, 152, &p)) {
      show(p);
      // the tile heights by themselves: the chosen plan's fields that none changes
      SimtPlan base = p, t;
      base.a.U2 = 0;
      base.a.G2 = base.a.two = 0;
      for (int c = 0; c < 4 && plan_tile(base, c, cap, 152, &t); ++c) show(t);
      // with a context's scratch: CTAs at work
      if (plan_simt(L, I, Q, KL, KQ, R, scratch_floats(L * Q, I, R, 152, true), 152, &p))
        printf(" %d %zu", p.grid, scratch_floats(L * Q, I, R, 152, true));
    }
    printf("\n");
  }
}
"""


@pytest.fixture(scope="module")
def planner(tmp_path_factory):
    d = tmp_path_factory.mktemp("plan")
    src, exe = d / "plan.cu", d / "plan"
    src.write_text(SOURCE)
    subprocess.run([build.nvcc_path(), "-std=c++17", "-O1", *build.ARCH, "-I" + build.CSRC,
                    "-I" + os.path.join(ROOT, "include"), str(src), "-o", str(exe)], check=True,
                   capture_output=True)
    return str(exe)


def _cases():
    r = random.Random(5)
    for _ in range(4000):
        N, R = r.randint(3, 5), r.randint(2, 128)
        d = [max(2, int(math.exp(r.uniform(math.log(8), math.log(500 if N == 3 else 80))))) for _ in range(N)]
        if r.random() < 0.2:
            d[r.randrange(N)] = r.randint(1000, 60000)
        lo = r.randint(0, N - 1)
        hi = lo + 1 if r.random() < 0.5 else r.choice([h for h in (lo + 1, N) if h - lo < N])
        if lo == 0 and r.random() < 0.5:
            hi = r.randint(1, N - 1)
        I = math.prod(d[lo:hi])
        tiles = -(-I // 128) * -(-R // 32)
        C = 1 if tiles >= 608 else min(-(-608 // tiles), max(1, -(-(math.prod(d) // I) // 256)))
        yield (N, R, lo, hi, r.choice([C * I * R if C > 1 else 0, 0, 1 << 21]), *d)
    # shapes whose largest tiles need no cut where smaller ones do
    yield (5, 42, 0, 3, 2159136, 18, 28, 51, 58, 11)
    yield (5, 68, 2, 5, 3366272, 44, 12, 14, 34, 52)


def test_every_tile_once_and_the_cheapest_height(planner):
    cases = list(_cases())
    out = subprocess.run([planner], input="\n".join(" ".join(map(str, c)) for c in cases) + "\n",
                         capture_output=True, text=True, check=True).stdout.splitlines()
    assert len(out) == len(cases)
    cut = 0
    for (N, R, lo, hi, cap, *d), line in zip(cases, out):
        v = [float(x) for x in line.split()]
        if not v:  # no tile fits: the ranks are then taken in blocks
            assert R > 8
            continue
        BM, whole, U2, nk, G2, two, grid, slot, cost = v[:9]
        I = math.prod(d[lo:hi])
        assert U2 % nk == 0 and whole + U2 // nk == -(-I // BM), (d, R, lo, hi)
        assert (G2 == 0) == (U2 == 0) and G2 <= grid and U2 >= G2
        assert (1 + two) * G2 * slot <= cap
        if not two and G2:
            assert G2 % (U2 // nk) == 0
        alone = [v[k:k + 9] for k in range(9, len(v) - 2, 9)]
        assert v[:9] in alone and cost == min(a[8] for a in alone), (d, R, lo, hi)
        cut += G2 > 0
        if I <= 512:  # few rows: 128 elements of the contraction per CTA, or a CTA per SM
            assert v[-2] >= min(150, nk // 4), (d, R, lo, hi)
        else:  # finer cuts of long outputs cost more in partial tiles than they save
            assert v[-1] == 0
    assert cut > 1000


@pytest.mark.parametrize("case", [(4, 8, 0, 2, 0, 4000, 21, 8, 14), (4, 3, 0, 3, 0, 59, 14, 56, 22)])
def test_few_steps_per_tile_take_one_split(planner, case):
    # the sums over a step's splits at the end of every tile would outweigh its few steps
    out = subprocess.run([planner], input=" ".join(map(str, case)) + "\n", capture_output=True, text=True,
                         check=True).stdout.split()
    assert float(out[0]) == 256
