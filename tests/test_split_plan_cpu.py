"""Schedule of the split FP64 FD's digit products (csrc/split_plan.h), as the
host compiler sees it: every step waits for the slices of B that it reads, the
steps hold every product of the kept groups once, and those of the leading
groups cannot pass the integers that FP32 accumulates exactly."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "..", "paper_1602_01636_gb300", "csrc")

PROGRAM = r"""
#include "split_plan.h"
#include <cstdio>
using namespace igafd_split;
template <int KP, int KT> void steps(int part) {
  for (int i = 0; i < Steps<KT>::kCount; ++i) {
    const Step s = Steps<KT>::at(i);
    printf("step %d %d %d %d %u %d %d %u\n", KP, part, KT, s.g, s.prods, s.k0, s.k1, step_waits(KP, s.g));
  }
}
template <int KP> void plan() {
  printf("first %d %d\n", KP, first_slices(KP));
  steps<KP, part_terms(KP)>(0);
  if constexpr (KP > part_terms(KP)) steps<KP, KP - part_terms(KP)>(1);
}
int main() {
  plan<32>(); plan<64>(); plan<96>(); plan<128>(); plan<160>(); plan<192>(); plan<224>(); plan<256>();
  printf("slices %d\n", kSlices);
}
"""


@pytest.fixture(scope="module")
def plan(tmp_path_factory):
    if not shutil.which("g++"):
        pytest.skip("no host compiler")
    d = tmp_path_factory.mktemp("plan")
    (d / "plan.cpp").write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-I", CSRC, str(d / "plan.cpp"), "-o", str(d / "plan")], check=True)
    out = subprocess.run([str(d / "plan")], check=True, capture_output=True, text=True).stdout
    first, steps, slices = {}, {}, 0
    for line in out.splitlines():
        kind, *v = line.split()
        v = [int(x) for x in v]
        if kind == "first":
            first[v[0]] = v[1]
        elif kind == "slices":
            slices = v[0]
        else:
            steps.setdefault((v[0], v[1], v[2]), []).append(v[3:])
    return first, steps, slices


def test_every_step_waits_for_the_slices_it_reads(plan):
    first, steps, slices = plan
    assert len(first) == 8 and slices == 6
    for (KP, _, _), todo in steps.items():
        for g, waits in ((s[0], s[-1]) for s in todo):
            for t in range(g + 1):                     # products of group g read slices 0 .. g of B
                assert waits >> (0 if t < first[KP] else 1) & 1, (KP, g, t)


def test_products_once_and_exact(plan):
    _, steps, slices = plan
    big = lambda s: 256 if s == 0 else 512             # 58 bits: 8 above five digits of 10
    for (_, _, KT), todo in steps.items():
        seen = []
        for g, prods, k0, k1, _ in todo:
            pairs = [(s, g - s) for s in range(slices) if prods >> s & 1]
            assert pairs and 0 <= k0 < k1 <= KT // 16
            seen += [(s, t, k) for s, t in pairs for k in range(k0, k1)]
            if g <= 3:
                assert 16 * (k1 - k0) * sum(big(s) * big(t) for s, t in pairs) <= 2 ** 24
        want = [(s, g - s, k) for g in range(slices) for s in range(g + 1) for k in range(KT // 16)]
        assert sorted(seen) == sorted(want)
