"""The host's scratch plan, called through the library's C++ functions."""

import os
import subprocess

import pytest

import paper_2605_29514_gb300 as stn
from paper_2605_29514_gb300 import _native

CHECK = r"""
#include <algorithm>
#include <cstdio>
#include <vector>
#include "engine.h"

int main() {
  int bad = 0;
  for (int n : {17, 49, 97, 161})
    for (int cap = 1; cap <= 256; ++cap) {
      std::vector<int> chi(n + 1, 1);
      for (int k = 1; k < n; ++k) chi[k] = std::min(cap, 1 << std::min({k, n - k, 20}));
      const stn::ScratchPlan full = stn::plan_scratch(n, chi.data(), cap);
      long long ap = 0, g = 0, c = *std::max_element(chi.begin(), chi.end());
      for (int k = 0; k < n; ++k) ap += 8ll * chi[k] * chi[k + 1];
      for (int k = 1; k < n; ++k) g += 4ll * chi[k] * chi[k];
      bad += full.ap_elems < ap || full.g_elems < g || full.work_elems < 35 * c * c + 4 * c + 1024;
      for (long long elems : {1ll << 40, ap + g, ap + g - 1, (ap + g) / 2 + 1, 12345ll, 1023ll, 17ll, 1ll, 0ll}) {
        stn::ScratchPlan p = full;
        stn::shrink_scratch(p, elems);
        for (int cta : {0, 1, 2, 303})  // of 8-byte elements: the CTA's share and its work area
          bad += 8 * (cta * p.total) % 16 != 0 || 8 * (cta * p.total + p.ap_elems + p.g_elems) % 16 != 0;
        bad += p.total != p.ap_elems + p.g_elems + p.work_elems || p.work_elems != full.work_elems;
        bad += p.ap_elems < 0 || p.g_elems < 0 || p.ap_elems + p.g_elems > elems;
        bad += elems >= ap + g && (p.ap_elems != ap || p.g_elems != g);
        const double f = std::min(1.0, static_cast<double>(elems) / (ap + g));
        bad += p.ap_elems + 4 < ap * f - 1 || p.g_elems + 4 < g * f - 1;
      }
    }
  std::printf("%d\n", bad);
  return bad != 0;
}
"""


def test_scratch_is_aligned_for_every_cap_and_arena(tmp_path):
    """Every CTA's share and its work area lie at multiples of 16 bytes in
    complex64, for every bond cap and for arenas that shrink the span stacks; a
    plan holds what it held, and a shrunk one at most the arena."""
    stn.build()
    src, exe = tmp_path / "check.cpp", tmp_path / "check"
    src.write_text(CHECK)
    cuda = os.path.dirname(os.path.dirname(_native.NVCC))
    subprocess.run(["g++", "-std=c++17", str(src), "-I", _native.CSRC, "-I", _native.INCLUDE, "-I", f"{cuda}/include",
                    _native.LIB, f"-L{cuda}/lib64", "-lcudart", f"-Wl,-rpath,{_native.PKG}:{cuda}/lib64", "-o", str(exe)],
                   check=True, capture_output=True, text=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
