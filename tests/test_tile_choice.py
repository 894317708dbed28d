"""The GEMM's tile rule (csrc/qlin_tiles.h, host code) at the sizes that its
comments quote, compiled and run on the CPU."""
import os
import shutil
import subprocess

import pytest

from conftest import ROOT

MAIN = r"""
#include <cstdio>
#include "qlin_tiles.h"
int main() {
  int kind, epi, sms; long long m, n, k;
  while (std::scanf("%d %d %lld %lld %lld %d", &kind, &epi, &m, &n, &k, &sms) == 6)
    std::printf("%d\n", (int)qlin::choose_tile((qlin::GemmKind)kind, (qlin::Epilogue)epi, m, n, k, sms));
}
"""
NVFP4, FP8, F16 = range(3)
PLAIN, REQUANT, AMAX = range(3)
PAIR, SINGLE, NARROW = range(3)


@pytest.fixture(scope="module")
def choose(tmp_path_factory):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    d = tmp_path_factory.mktemp("tiles")
    (d / "main.cpp").write_text(MAIN)
    csrc = os.path.join(ROOT, "paper_2609_21849_gb300", "csrc")
    subprocess.run([cxx, "-std=c++17", "-I" + csrc, str(d / "main.cpp"), "-o", str(d / "main")],
                   check=True)

    def run(cases):
        text = "".join("%d %d %d %d %d 152\n" % c for c in cases)
        out = subprocess.run([str(d / "main")], input=text, capture_output=True, text=True, check=True)
        return [int(v) for v in out.stdout.split()]
    return run


def test_quoted_sizes(choose):
    want = {
        # the fitted times against the counts: fewer pair tiles than SMs, but the
        # single ones' last wave is nearly empty; K too short for pairs
        (NVFP4, PLAIN, 1000, 3072, 3072): PAIR,
        (NVFP4, PLAIN, 4608, 2560, 256): SINGLE,
        (NVFP4, PLAIN, 18432, 1024, 64): SINGLE,
        # within the margin: the count decides
        (NVFP4, PLAIN, 3000, 3072, 256): PAIR,
        (FP8, PLAIN, 3000, 3072, 256): PAIR,
        (F16, PLAIN, 3000, 3072, 256): PAIR,
        # an output amax keeps the pair tiles at short K, fused and plain do not
        (NVFP4, AMAX, 9216, 3072, 64): PAIR,
        (NVFP4, AMAX, 9216, 2560, 64): PAIR,
        (NVFP4, AMAX, 4608, 12288, 256): PAIR,
        (NVFP4, AMAX, 129, 9984, 704): SINGLE,
        (NVFP4, PLAIN, 9216, 3072, 64): SINGLE,
        (NVFP4, REQUANT, 4608, 12288, 256): SINGLE,
        (NVFP4, AMAX, 1000, 3072, 3072): PAIR,
        # the large layers and the translator's
        (NVFP4, REQUANT, 4608, 12288, 3072): PAIR,
        (NVFP4, AMAX, 4608, 9216, 3072): PAIR,
        (FP8, PLAIN, 4608, 3072, 3072): PAIR,
        (F16, PLAIN, 4608, 3072, 3072): PAIR,
        (NVFP4, REQUANT, 512, 2560, 3072): SINGLE,
        (NVFP4, PLAIN, 512, 1024, 2560): NARROW,
        (NVFP4, REQUANT, 512, 1024, 2560): SINGLE,
        (F16, PLAIN, 512, 1024, 2560): SINGLE,
    }
    got = choose(want)
    assert got == list(want.values()), [(c, g) for (c, w), g in zip(want.items(), got) if w != g]
