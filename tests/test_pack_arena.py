"""The shared-memory arena of a packed launch: as many CTAs as the grid counts on fit an SM together, with
each one's static shared memory and the system's share (228 KB an SM, 227 KB a CTA, 1 KB each for the
system, allocated by 128 bytes)."""
import os
import subprocess

import pytest

from tests._lib import ROOT

PROGRAM = r"""
#include <cstdio>
#include "batch.h"
int main() {
  for (int per_sm : {1, 2, 3, 4})
    for (int tab : {0, 17, 700, tn::kMaxTabInts})
      for (long long largest : {0ll, 64ll, 4096ll, 20000ll, 1ll << 30})
        std::printf("%d %d %lld %d %d\n", per_sm, tab, largest, tn::pack_arena_floats(per_sm, tab, largest),
                    tn::kBatchStaticSmem);
}
"""


def test_ctas_fit_together(tmp_path):
    src, exe = tmp_path / "arena.cpp", tmp_path / "arena"
    src.write_text(PROGRAM)
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    if not os.path.exists(os.path.join(cuda, "include", "cuda_runtime.h")):
        pytest.skip("no CUDA headers")
    subprocess.run(["g++", "-std=c++17", "-I", os.path.join(ROOT, "paper_2606_01852_gb300", "csrc"), "-I",
                    os.path.join(cuda, "include"), str(src), "-o", str(exe)], check=True)
    lines = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split("\n")
    for line in filter(None, lines):
        per_sm, tab, largest, arena, static = map(int, line.split())
        dynamic = 4 * (arena // 64 * 64 + tab)
        cta = (dynamic + static + 127) // 128 * 128
        assert cta <= 227 * 1024 and per_sm * (cta + 1024) <= 228 * 1024
        assert arena <= largest
        # and less than 1 KB a CTA is given away
        assert arena == largest or per_sm * (cta + 1024 + 1024) > 228 * 1024
