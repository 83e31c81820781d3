"""Slot counts of the stream-K plan, on the CPU: a small host program asks the built library for plans and compares the reciprocal
arithmetic that the consumer kernels use with plain divisions, tile by tile."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
PKG = os.path.join(ROOT, "paper_2402_05109_b200")

PROGRAM = r"""
#include "launch.h"
#include <cstdio>
#include <cstdlib>
using namespace hydra;
int main() {
  const int shapes[][3] = {{1, 128, 64}, {1, 128, 128}, {64, 4096, 4096}, {128, 22016, 4096}, {257, 4096, 11008}, {768, 32000, 4096}, {4096, 32000, 6656},
                           {29975, 37888, 50432}, {57707, 37760, 35328}, {40000000, 128, 64}, {20000001, 256, 64}};      // far past what a model asks for
  for (auto& s : shapes) {
    const SplitDesc sd = gemm_tc_plan(s[0], s[1], s[2], nullptr, nullptr);
    const int step = s[0] > 1000000 ? 9973 : 1;
    for (long long n = 0; n < s[1]; n += 1 << sd.bn_shift)
      for (long long t = 0; t < sd.m_tiles; t += step)
        for (long long m : {t * sd.mt, std::min<long long>((t + 1) * sd.mt, s[0]) - 1}) {
          const long long u0 = ((n >> sd.bn_shift) * sd.m_tiles + m / sd.mt) * sd.kb, want = (u0 + sd.kb - 1) / sd.q - u0 / sd.q + 1;
          if (split_count(sd, (int)m, (int)n) != want) return printf("%d x %d x %d: row %lld column %lld\n", s[0], s[1], s[2], m, n), 1;
        }
  }
  unsigned long long r = 88172645463325252ull;             // xorshift
  auto rnd = [&](unsigned below) { r ^= r << 13; r ^= r >> 7; r ^= r << 17; return (unsigned)((r >> 16) % below); };
  for (int i = 0; i < 2000000; ++i) {
    SplitDesc sd{};
    sd.q = 1 + (int)rnd(1u << (1 + rnd(31))); sd.mt = 16; sd.m_tiles = 1;
    sd.set_inverses();
    const unsigned near = rnd(0x7fffffffu / (unsigned)sd.q + 1) * (unsigned)sd.q;          // a multiple of q and its neighbours
    for (unsigned u : {near, near ? near - 1 : 0u, rnd(0x7fffffffu)})
      if (sd.div_q(u) != u / (unsigned)sd.q) return printf("%u / %d\n", u, sd.q), 1;
  }
  const SplitDesc one = single_slot(0);
  return split_count(one, 4095, 151935) == 1 ? 0 : 2;
}
"""


def test_slot_counts_against_divisions(tmp_path):
    from paper_2402_05109_b200.build import build
    build()
    src, exe = tmp_path / "plan.cu", tmp_path / "plan"
    src.write_text("#include <algorithm>\n#include <initializer_list>\n" + PROGRAM)
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    subprocess.run([nvcc, "-gencode", "arch=compute_100a,code=sm_100a", "-std=c++17", "-O2", "-I", os.path.join(PKG, "csrc"), str(src), "-o", str(exe),
                    "-L", PKG, "-lhydra", "-Xlinker", "-rpath=" + PKG], check=True, capture_output=True, text=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout
