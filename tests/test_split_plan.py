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


ERRORS = r"""
#include "launch.h"
#include <cstdio>
#include <cmath>
using namespace hydra;
// Error of a product by its plan, up to a factor: sums are drained where a range or a tile ends, and an error grows with a sum's length to the power 1.5.
static double error(long long line, int kb, int q) {
  double s = 0;
  for (long long u = 0; u < line;) {
    const long long end = std::min({(u / kb + 1) * kb, (u / q + 1) * q, line});
    s += std::pow((double)(end - u), 3);
    u = end;
  }
  return std::sqrt(s / (double)line);
}
int main() {
  const int shapes[][2] = {{4096, 4096}, {12288, 4096}, {22016, 4096}, {4096, 11008}, {32000, 4096}, {5120, 5120}, {5120, 13824}, {6656, 6656}, {35840, 6656}, {6656, 17920},
                           {2048, 2048}, {1024, 1024}, {3072, 1024}, {4224, 2048}};
  int bad = 0;
  for (auto& s : shapes)
    for (int tiles = 2; tiles <= 64; ++tiles) {
      const int n = s[0], k = s[1], m = 256 * tiles - 16, kb = k / 64;      // row tiles of 256
      int grid = 0;
      const SplitDesc sd = gemm_tc_plan(m, n, k, &grid, nullptr);
      const long long n_tiles = (n + (1 << sd.bn_shift) - 1) >> sd.bn_shift, all = n_tiles * tiles * kb, sms = sm_count();
      if (all / 4 < sms) continue;
      const int q1 = (int)((all + sms - 1) / sms);
      const double one = error(all, kb, q1), now = error(n_tiles * sd.m_tiles * kb, kb, sd.q);
      if (now > 1.051 * one || 8ll * sd.q > 9ll * q1 || grid > sms) ++bad, printf("%d row tiles of %d x %d: error %.3f, ranges %d / %d, grid %d\n", tiles, n, k, now / one, sd.q, q1, grid);
    }
  return bad != 0;
}
"""


def test_row_tiles_that_walk_together_have_sums_as_short_as_alone(tmp_path):
    from paper_2402_05109_b200.build import build
    build()
    src, exe = tmp_path / "errors.cu", tmp_path / "errors"
    src.write_text("#include <algorithm>\n#include <initializer_list>\n" + ERRORS)
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    subprocess.run([nvcc, "-gencode", "arch=compute_100a,code=sm_100a", "-std=c++17", "-O2", "-I", os.path.join(PKG, "csrc"), str(src), "-o", str(exe),
                    "-L", PKG, "-lhydra", "-Xlinker", "-rpath=" + PKG], check=True, capture_output=True, text=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout
