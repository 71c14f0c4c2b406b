"""The words that the stem kernel's gather threads request (csrc/stem_words.h), enumerated on the host: a read past the image
batch cannot be seen by guards around a buffer, which only catch writes."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

# every image row, filter row and output pixel of a batch: the requested words lie in the batch, and hold every element of the run that
# lies in the row
HARNESS = r"""
#include "stem_words.h"
#include <cstdio>
#include <cstdlib>
#include <initializer_list>
static void fail(const char* what, int kh, int B, int H, int W, long at) {
  std::printf("%s: %dx%d filter, B %d, H %d, W %d, element %ld\n", what, kh, kh, B, H, W, at);
  std::exit(1);
}
int main() {
  long words = 0, odd = 0, alone = 0;
  for (int kh : {7, 3}) {
    const int pad = kh / 2, NW = (1 + kh * 3 + 1) / 2;
    for (int B = 1; B <= 4; ++B)
      for (int H : {1, 2, 3, 5})
        for (int W = 1; W <= 257; ++W) {
          const int Wo = (W - 1) / 2 + 1, row = W * 3;
          if (Wo > 128) continue;
          const long total = (long)B * H * row;
          for (int n = 0; n < B; ++n)
            for (int y = 0; y < H; ++y)
              for (int ox = 0; ox < Wo; ++ox) {
                const int e0 = 6 * ox - 3 * pad - 1;
                const long rb = ((long)n * H + y) * row;
                const ee::StemTaps t = ee::stem_taps(e0, row, NW);
                const ee::StemAsk a = ee::stem_ask(rb, row, total, t);
                bool have[2 * 16 + 4] = {};   // element e0 - 1 + i of the row is loaded
                for (int j = 0; j < NW + (a.kind == 2 ? 1 : 0); ++j) {
                  if (!(a.mask >> j & 1u)) continue;
                  const int e = e0 + a.off + 2 * j;
                  if ((rb + e) & 1) fail("unaligned word", kh, B, H, W, rb + e);
                  if (rb + e < 0 || rb + e + 2 > total) fail("word outside the batch", kh, B, H, W, rb + e);
                  have[e - e0 + 1] = have[e - e0 + 2] = true;
                  ++words;
                }
                if (a.mask >> (NW + (a.kind == 2 ? 1 : 0))) fail("a word that no register takes", kh, B, H, W, rb);
                if (a.kind == 3 && t.first && row - 1 >= e0 && row - 1 - e0 + 1 < 36) have[row - 1 - e0 + 1] = true, ++alone;
                odd += a.kind == 2;
                for (int i = 0; i < 2 * NW; ++i)
                  if (e0 + i >= 0 && e0 + i < row && !have[i + 1]) fail("element not loaded", kh, B, H, W, rb + e0 + i);
              }
        }
  }
  std::printf("%ld words, %ld odd rows, %ld single elements\n", words, odd, alone);
  return !(words && odd && alone);
}
"""


def test_requested_words_lie_in_the_batch_and_hold_the_run(tmp_path):
    src, exe = tmp_path / "words.cpp", tmp_path / "words"
    src.write_text(HARNESS)
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", os.path.join(ROOT, "paper_2209_13443_b200", "csrc"), "-o", str(exe), str(src)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout


# a thread per pixel pair: three words from element 6 r of every image row on, and what of them is read
PAIRS = r"""
#include "stem_words.h"
#include <cstdio>
#include <initializer_list>
int main() {
  long halves = 0, odd = 0;
  for (int B = 1; B <= 3; ++B)
    for (int H : {1, 2, 3, 5})
      for (int W = 1; W <= 256; ++W) {
        const int Wo = (W - 1) / 2 + 1, row = W * 3;
        const long total = (long)B * H * row;
        for (long y = 0; y < (long)B * H; ++y)
          for (int r = 0; r < Wo; ++r) {
            const ee::StemTaps in = ee::stem_taps(6 * r, row, 3);
            const ee::StemAsk a = ee::stem_ask(y * row, row, total, in);
            bool have[10] = {};   // element 6 r - 1 + i of the row
            for (int j = 0; j <= 3; ++j) {
              const int n = ee::stem_word_bytes(a, in, j);
              if (j == 3 && a.kind != 2 && n) return std::printf("a fourth word of an even row\n"), 1;
              const long e = y * row + 6 * r + a.off + 2 * j;
              if (n && ((e & 1) || e < 0 || e + n / 2 > total)) return std::printf("B %d H %d W %d: %d bytes at element %ld of %ld\n", B, H, W, n, e, total), 1;
              for (int i = 0; i < n / 2; ++i) have[1 + a.off + 2 * j + i] = true;
              halves += n == 2;
            }
            odd += a.kind == 2;
            for (int i = 0; i < 6; ++i)
              if (6 * r + i < row && !have[1 + i]) return std::printf("B %d H %d W %d: element %d of pair %d not read\n", B, H, W, i, r), 1;
          }
      }
  return !(halves && odd);
}
"""


def test_pixel_pairs_are_read_whole_and_inside_the_batch(tmp_path):
    src, exe = tmp_path / "pairs.cpp", tmp_path / "pairs"
    src.write_text(PAIRS)
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", os.path.join(ROOT, "paper_2209_13443_b200", "csrc"), "-o", str(exe), str(src)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
