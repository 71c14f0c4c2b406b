"""How an exit head's FC layer is cut over CTAs (csrc/fc_shape.h): which heads the cluster kernel takes, and that every tile of
every batch fits its shared memory, the counters and the exchange buffer."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

HARNESS = r"""
#include "fc_shape.h"
#include <cstdio>
#include <initializer_list>
#define NEED(c) if (!(c)) { std::printf("%s: %d-byte weights, C %d, K %d, B %d, room %d\n", #c, es, C, K, B, room); return 1; }
int main() {
  int B = 0, room = 0, es = 0, C = 0, K = 0;
  // heads on more channels, and with more classes, than a tile of eight samples has shared memory for
  for (int e : {2, 4}) {
    es = e;
    for (int c : {2048, 2816, 3072, 4096, 8192, 16384}) { C = c; K = 1000; NEED(ee::fc_fits(C, K, es)); }
    for (int k : {10, 1000, 16000, 22000, 90000}) { C = 512; K = k; NEED(ee::fc_fits(C, K, es)); }
  }
  int capped = 0;
  for (int e : {2, 4})
    for (int c : {8, 512, 2048, 2816, 3072, 4096, 6144, 8192, 12288, 16384, 24064, 24320, 32768})
      for (int k : {2, 10, 64, 65, 512, 513, 1000, 5000, 22000, 90000, 400000}) {
        es = e, C = c, K = k;
        if (!ee::fc_fits(C, K, es)) continue;
        const ee::FcShape one = ee::fc_shape(1, C, K, es, 4);
        for (int r : {1, 4, 7})
          for (B = 1; B <= 80; ++B) {
            room = r;
            const ee::FcShape f = ee::fc_shape(B, C, K, es, room);
            NEED(ee::fc_smem_bytes(f) <= (size_t)ee::kFcMaxSmem);
            NEED(f.CL == one.CL && f.kb == one.kb && f.Cp == one.Cp);   // what fixes a sum does not depend on the batch
            NEED((f.S & (f.S - 1)) == 0 && f.S >= 1 && f.S <= (es == 4 ? 4 : 8));
            const long tiles = (B + f.S - 1) / f.S;
            NEED(tiles <= B);                                           // a counter per sample of max_batch
            // without clusters the blocks' triples lie where the batch's logits do
            if (!f.cluster && f.CL > 1) NEED(tiles * ee::kFcBlocks * f.S * 16 <= (long)B * K * 4);
            capped += f.S < ee::fc_shape(B, 8, 8, es, room).S;
          }
      }
  return !capped;
}
"""


def test_wide_heads_are_taken_and_every_tile_fits(tmp_path):
    src, exe = tmp_path / "shape.cpp", tmp_path / "shape"
    src.write_text(HARNESS)
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", os.path.join(ROOT, "paper_2209_13443_b200", "csrc"), "-o", str(exe), str(src)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout


# models of few samples: at least eight CTAs for many channels, warps that share a class's channels; the cut does not depend on the batch
SHARED = r"""
#include "fc_shape.h"
#include <cstdio>
#include <initializer_list>
#define NEED(c) if (!(c)) { std::printf("%s: %d-byte weights, C %d, K %d, B %d of %d\n", #c, es, C, K, B, most); return 1; }
int main() {
  int shared = 0, deep = 0, B = 1;
  for (int es : {2, 4})
    for (int most : {1, 6, 32, 33})
      for (int C : {4, 128, 512, 2048, 8192, 24064})
        for (int K : {1, 10, 64, 100, 129, 1000}) {
          if (C * es % 16 || !ee::fc_fits(C, K, es)) continue;
          const ee::FcShape one = ee::fc_shape(1, C, K, es, 4, most);
          const int nchunk = one.Cp * es / 512, groups = ee::kFcBlocks / one.CL * one.kb / ee::kFcRows;
          NEED(one.ws >= 1 && one.ws <= nchunk && (one.ws == 1 || one.ws * groups <= ee::kFcThreads / 32));   // every warp has a slot
          NEED(most > 32 || nchunk < 4 || one.CL >= 8);
          for (B = 1; B <= most; ++B) {
            const ee::FcShape f = ee::fc_shape(B, C, K, es, 4, most);
            NEED(f.CL == one.CL && f.ws == one.ws && f.kb == one.kb);
            NEED(f.ring >= 2 && f.ring <= 6 && ee::fc_smem_bytes(f) <= (size_t)ee::kFcMaxSmem);
            NEED(!ee::fc_pools(f, 33, 32) && (!ee::fc_pools(f, 32, 32) || (f.CL == 1 && f.S == 1)));
            shared += f.ws > 1, deep += f.ring == 6;
          }
        }
  return !(shared && deep);
}
"""


def test_warps_that_share_channels(tmp_path):
    src, exe = tmp_path / "shared.cpp", tmp_path / "shared"
    src.write_text(SHARED)
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", os.path.join(ROOT, "paper_2209_13443_b200", "csrc"), "-o", str(exe), str(src)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
