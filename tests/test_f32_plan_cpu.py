"""Tile and K cut of the fp32 model's convolutions (csrc/f32_plan.h): every CTA of a cluster has work, and about the same."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

HARNESS = r"""
#include "f32_plan.h"
#include <cstdio>
#include <initializer_list>
int main() {
  int cut = 0;
  for (int k = 1; k <= 12000; ++k)
    for (long m : {1L, 16L, 24L, 32L, 96L, 400L, 1536L, 6000L, 100000L})
      for (int n : {8, 64, 128, 512, 2048}) {
        const ee::F32Plan p = ee::f32_plan(m, n, k, 148);
        const int per = ee::f32_k_per(k, p.z);
        int covered = 0, most = 0, least = k;
        for (int z = 0; z < p.z; ++z) {
          const int lo = z * per, hi = lo + per < k ? lo + per : k, len = hi - lo;
          if (len <= 0) { std::printf("K %d, M %ld, N %d: CTA %d of %d has no work\n", k, m, n, z, p.z); return 1; }
          covered += len;
          most = len > most ? len : most, least = len < least ? len : least;
        }
        // unequal by at most the rounding of K to 16 and of the steps to the CTAs
        if (covered != k || per % 16 || (p.z > 1 && most - least >= 16 * p.z)) { std::printf("K %d, M %ld, N %d: %d to %d over %d CTAs\n", k, m, n, least, most, p.z); return 1; }
        cut += p.z > 1;
      }
  return !cut;
}
"""


def test_every_cta_of_a_cluster_has_work(tmp_path):
    src, exe = tmp_path / "plan.cpp", tmp_path / "plan"
    src.write_text(HARNESS)
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", os.path.join(ROOT, "paper_2209_13443_b200", "csrc"), "-o", str(exe), str(src)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout


LINES = r"""
#include "f32_plan.h"
#include <cstdio>
#include <initializer_list>
int main() {
  int seen[4] = {0, 0, 0, 0}, cut = 0;
  for (bool vec : {true, false})
    for (int k = 1; k <= 12000; ++k)
      for (long m : {1L, 16L, 17L, 32L, 33L, 96L, 400L, 1536L, 6000L, 100000L})
        for (int n : {1, 8, 33, 64, 512, 2048}) {
          const ee::F32Plan p = ee::f32_plan(m, n, k, 148, vec);
          const int per = ee::f32_k_per(k, p.z);
          const bool short_k = k < (vec ? 128 : 256);
          const char* wrong = short_k != (p.tile == 0)                     ? "one K group for short K alone"
                              : p.tile < 2 && p.z != 1                     ? "a tile that receives nothing is cut"
                              : (p.tile == 3) != (p.tile >= 2 && m <= 32)  ? "16 rows up to 32 of them"
                              : p.z & (p.z - 1) || p.z > 8                 ? "1, 2, 4 or 8 CTAs"
                              : p.z > 1 && per < 64                        ? "less than 64 of K"
                              : (p.z - 1L) * per >= k                      ? "a CTA without work"
                                                                           : nullptr;
          if (wrong) { std::printf("K %d, M %ld, N %d, vec %d: tile %d, %d CTAs: %s\n", k, m, n, vec, p.tile, p.z, wrong); return 1; }
          ++seen[p.tile], cut += !vec && p.z > 1;
        }
  return !(seen[0] && seen[1] && seen[2] && seen[3] && cut);
}
"""


def test_lines_of_the_plan_with_copies_of_16_and_of_4_bytes(tmp_path):
    src, exe = tmp_path / "lines.cpp", tmp_path / "lines"
    src.write_text(LINES)
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", os.path.join(ROOT, "paper_2209_13443_b200", "csrc"), "-o", str(exe), str(src)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
