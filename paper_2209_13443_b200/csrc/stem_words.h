// Which 32-bit words of an image row a gather thread of the stem kernel (conv_stem.cuh) asks for.  Plain arithmetic, for the
// device and for host tests: a word is two bf16 elements of an image batch whose end is the end of the caller's buffer.
#pragma once
#include <stdint.h>

#ifdef __CUDACC__
#define EE_HD __host__ __device__ __forceinline__
#else
#define EE_HD inline
#endif

namespace ee {

// A filter row's run in an image row: elements e0, e0 + 1, ... of the row, e0 even (negative left of the image).
// Bit j of `first` / `second`: element e0 + 2 j / e0 + 2 j + 1 lies inside the row.
struct StemTaps {
  uint32_t first, second;
};
EE_HD StemTaps stem_taps(int e0, int row_elems, int words) {
  StemTaps t = {0u, 0u};
#pragma unroll
  for (int j = 0; j < words; ++j) {
    t.first |= (e0 + 2 * j >= 0 && e0 + 2 * j < row_elems ? 1u : 0u) << j;
    t.second |= (e0 + 2 * j >= 0 && e0 + 2 * j + 1 < row_elems ? 1u : 0u) << j;
  }
  return t;
}

// The aligned words to load for a row that begins at element row_begin of the batch's `total`: bit j of `mask` = the word of
// the elements e0 + off + 2 j and e0 + off + 2 j + 1.
//   kind 0: the row begins at an even element; words and run coincide.
//   kind 2: it begins at an odd one (rows of an odd number of elements): word j holds run elements 2 j - 1 and 2 j, and is
//           loaded if either lies in the row.  Its other half is then in the batch: a row's elements from an odd one on
//           end at an even one, and in front of an odd row there is another.
//   kind 3: even, but the row's last element is the batch's last and alone in its word: that word is left out, the element
//           is loaded by itself.
struct StemAsk {
  int kind, off;
  uint32_t mask;
};
EE_HD StemAsk stem_ask(long row_begin, int row_elems, long total, StemTaps t) {
  StemAsk a;
  if (row_begin & 1) {
    a.kind = 2, a.off = -1, a.mask = t.first | t.second << 1;
  } else {
    a.kind = (row_elems & 1) && row_begin + row_elems == total ? 3 : 0;
    a.off = 0, a.mask = a.kind == 3 ? t.second : t.first;
  }
  return a;
}
// Bytes of word j that are read, from element e0 + off + 2 j on: 4, 2 (kind 3: the batch's last element, alone in its word) or none.
EE_HD int stem_word_bytes(StemAsk a, StemTaps in, int j) {
  if (a.mask >> j & 1u) return 4;
  return a.kind == 3 && ((in.first & ~in.second) >> j & 1u) ? 2 : 0;
}

}  // namespace ee
