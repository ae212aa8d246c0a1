"""Launch shapes of the symmetric-storage substitution (csrc/hd_sym_shape.cuh, plain host code):
every shape can serve the launch it is picked for, and the picks are the fastest, or within a few
per cent of it, of the forms measured on the GPU (152 SMs)."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1508_02897_gb300", "csrc")
SMS = 152

HARNESS = r"""
#include <cstdio>
#include "hd_sym_shape.cuh"
int main() {
  int f, m, nrhs, sms;
  long nsub;
  while (std::scanf("%d %d %ld %d %d", &f, &m, &nsub, &nrhs, &sms) == 5) {
    const hd::SymPick p = f ? hd::sym_pick64(m, nsub, nrhs, sms) : hd::sym_pick32(m, nsub, nrhs, sms);
    std::printf("%d %d %d %d %d\n", p.K, p.P, p.SW, p.NR, p.per_sm);
  }
}
"""


@pytest.fixture(scope="module")
def picks(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("needs a C++ compiler")
    d = tmp_path_factory.mktemp("shape")
    (d / "shape.cpp").write_text(HARNESS)
    exe = str(d / "shape")
    subprocess.run([cxx, "-std=c++17", "-O1", "-I", CSRC, str(d / "shape.cpp"), "-o", exe], check=True)

    def run(cases):
        text = "".join("%d %d %d %d %d\n" % c for c in cases)
        out = subprocess.run([exe], input=text, capture_output=True, text=True, check=True).stdout
        return [tuple(map(int, line.split())) for line in out.splitlines()]
    return run


@pytest.mark.parametrize("fp64", [0, 1])
def test_every_pick_can_serve_its_launch(picks, fp64):
    cases = [(fp64, m, b, q, sms) for m in range(1, 257) for b in (1, 3, 38, 39, 76, 77, 152, 153, 305, 2000)
             for q in (1, 2, 3, 4, 5, 9) for sms in (1, 148, SMS)]
    for (_, m, b, q, sms), (K, P, SW, NR, per_sm) in zip(cases, picks(cases)):
        mp = (m + 15) // 16 * 16
        assert 32 * P * SW >= mp                      # a thread per row of the widest box
        assert K in (1, 2, 4) and K * P in (1, 2, 4)  # the four groups of segments divide
        assert NR in ((1,) if fp64 else (1, 2, 4)) and NR < 2 * q
        assert per_sm * (P * SW + 1) * 32 <= 1024
        # the compiled forms
        forms = ((1, 1, 3, 4), (1, 1, 4, 3), (1, 1, 8, 1), (1, 1, 8, 2), (2, 1, 8, 1), (4, 1, 8, 1)) if fp64 else \
            ((1, 1, 3, 4), (4, 1, 7, 1), (2, 2, 7, 1), (1, 2, 7, 1))
        assert (K, P, SW, per_sm) in forms


SMALL, MID = (1, 1, 3, 4), (1, 1, 4, 3)   # K, P, SW, CTAs per SM

# complex FP64?, widest box, boxes, sources, the forms (K, P, SW, per SM) and sources per CTA that were
# measured as fastest or within 5 % of it
MEASURED = [
    (0, 20, 256, 1, [SMALL + (1,)]), (0, 32, 1024, 1, [SMALL + (1,)]), (0, 48, 400, 1, [SMALL + (1,)]),
    (0, 64, 4096, 1, [SMALL + (1,)]), (0, 96, 1024, 1, [SMALL + (1,)]), (0, 64, 1024, 4, [SMALL + (4,)]),
    (0, 64, 256, 4, [SMALL + (2,)]), (0, 64, 256, 2, [SMALL + (1,)]), (0, 64, 144, 4, [SMALL + (1,)]),
    (0, 64, 144, 1, [(1, 2, 7, 1, 1)]), (0, 64, 64, 1, [(2, 2, 7, 1, 1)]), (0, 64, 4, 4, [(4, 1, 7, 1, 1)]),
    (0, 112, 1024, 1, [(1, 2, 7, 1, 1)]), (0, 176, 16, 1, [(4, 1, 7, 1, 1)]), (0, 176, 64, 1, [(2, 2, 7, 1, 1)]),
    (0, 176, 1024, 1, [(1, 2, 7, 1, 1)]), (0, 176, 256, 4, [(1, 2, 7, 1, 4)]), (0, 256, 4, 1, [(2, 2, 7, 1, 1)]),
    (1, 20, 256, 1, [SMALL + (1,)]), (1, 32, 1024, 2, [SMALL + (1,)]), (1, 48, 169, 1, [SMALL + (1,)]),
    (1, 80, 400, 1, [SMALL + (1,)]), (1, 64, 256, 1, [(1, 1, 8, 2, 1)]), (1, 64, 100, 1, [(1, 1, 8, 1, 1)]),
    (1, 64, 64, 1, [(2, 1, 8, 1, 1)]), (1, 96, 100, 1, [(1, 1, 8, 1, 1)]), (1, 96, 169, 1, [(1, 1, 8, 2, 1)]),
    (1, 112, 36, 1, [(4, 1, 8, 1, 1)]), (1, 112, 100, 1, [(1, 1, 8, 1, 1)]), (1, 112, 169, 1, [(2, 1, 8, 1, 1)]),
    (1, 112, 256, 2, [(1, 1, 8, 2, 1)]), (1, 112, 400, 1, [MID + (1,)]), (1, 144, 100, 1, [(1, 1, 8, 1, 1)]),
    (1, 176, 64, 1, [(2, 1, 8, 1, 1)]), (1, 176, 100, 1, [(1, 1, 8, 1, 1)]), (1, 240, 64, 2, [(1, 1, 8, 1, 1)]),
    (1, 240, 100, 1, [(4, 1, 8, 1, 1)]), (1, 240, 169, 1, [(4, 1, 8, 1, 1)]),
]


def test_picks_are_the_measured_ones(picks):
    got = picks([c[:4] + (SMS,) for c in MEASURED])
    for (fp64, m, b, q, good), (K, P, SW, NR, per_sm) in zip(MEASURED, got):
        assert (K, P, SW, per_sm, NR) in good, (fp64, m, b, q, (K, P, SW, per_sm, NR))
