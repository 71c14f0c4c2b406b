"""Which tensor maps a launch of a tensor-core convolution builds and keeps (csrc/conv_tc.cuh): host code, run without a GPU."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
NVCC = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")

# The launches themselves fail or do nothing without a GPU; what counts is what they left in the layer's cache.
HARNESS = r"""
#include <algorithm>
#include <cstdio>
#include <string>
#include <vector>
#include "common.cuh"
#include "conv_tc.cuh"
#include "conv_wave.cuh"
using namespace ee;
static CUresult tiled(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                      CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill) { return CUDA_SUCCESS; }
static CUresult im2col(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*, const int*, const int*, cuuint32_t, cuuint32_t,
                       const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill) { return CUDA_SUCCESS; }
static TcContext ctx;
static TcLayer layer(int hw, int cin, int cout, int k, int most) {
  ee_layer_desc_t d = {};
  d.op = EE_OP_CONV, d.cin = cin, d.cout = cout, d.kh = d.kw = k, d.stride = 1, d.pad = d.pad_w = k / 2;
  TcLayer L;
  tc_plan_layer(ctx, d, hw, hw, hw, hw, most, nullptr, &L);
  return L;
}
static std::string kinds(const TcLayer& L) {
  std::vector<int> k;
  for (const auto& e : L.a_maps) k.push_back(e.kind);
  std::sort(k.begin(), k.end());
  std::string r;
  for (int v : k) r += (r.empty() ? "" : ",") + std::to_string(v);
  return r;
}
static int bad(const char* what, const TcLayer& L, const std::string& want) {
  if (kinds(L) == want) return 0;
  std::printf("%s: maps of kinds %s, not %s\n", what, kinds(L).c_str(), want.c_str());
  return 1;
}
int main() {
  ctx.encode_tiled = tiled, ctx.encode_im2col = im2col, ctx.sm_count = 148;
  alignas(64) static char buf[32768];
  const void *x = buf + 4096, *r = buf + 8192;
  void* y = buf + 16384;
  int e = 0;
  auto run = [&](const TcLayer& L, int B, bool res, int mode = 0) { tc_launch(ctx, L, x, res ? r : nullptr, y, B, nullptr, nullptr, nullptr, 0, nullptr, 0, mode); };
  { TcLayer L = layer(7, 512, 512, 3, 64); run(L, 1, false); e += bad("64-pixel tiles", L, "9"); run(L, 1, false); e += bad("the same call again", L, "9"); }
  { TcLayer L = layer(14, 256, 1024, 1, 64); run(L, 1, true); e += bad("one wave, residual", L, "9"); }
  { TcLayer L = layer(14, 256, 512, 3, 64); run(L, 20, false); e += bad("128-pixel tiles in one wave", L, "0"); }
  { TcLayer L = layer(56, 64, 256, 1, 64); run(L, 64, true); e += bad("persistent, residual", L, "0,7,8"); }
  { TcLayer L = layer(56, 256, 64, 1, 64); run(L, 64, false); e += bad("persistent", L, "0,8"); }
  { TcLayer L = layer(28, 128, 128, 3, 64); run(L, 64, true); e += bad("several waves, residual", L, "0,1,7"); }
  { TcLayer L = layer(7, 512, 512, 3, 64); tc_set_splits(L, 4); run(L, 1, true, 1); e += bad("clusters of ranges", L, "0"); }
  { TcLayer L = layer(7, 512, 512, 3, 64); tc_set_splits(L, 4); run(L, 64, true, 2); e += bad("ranges in one CTA", L, "0,1,7"); }
  for (int B : {1, 64}) {
    TcLayer L = layer(56, 64, 256, 1, 64), P = layer(56, 64, 256, 1, 64);
    tc_launch_proj(ctx, L, P, x, r, y, B, nullptr, nullptr, nullptr, nullptr, nullptr, 0);
    e += bad("projection inside", L, B == 1 ? "0" : "0,8") + bad("projection", P, "0");
  }
  return e != 0;
}
"""


@pytest.mark.skipif(not (os.path.exists(NVCC) or shutil.which(NVCC)), reason="needs nvcc")
def test_a_launch_keeps_the_maps_its_kernel_reads_and_no_others(tmp_path):
    src, exe = tmp_path / "maps.cu", tmp_path / "maps"
    src.write_text(HARNESS)
    inc = [os.path.join(ROOT, "paper_2209_13443_b200", "csrc"), os.path.join(ROOT, "include")]
    # PTX is not assembled: the kernels never run
    subprocess.run([NVCC, "-std=c++17", "-O0", "-gencode", "arch=compute_100a,code=compute_100a"] + [f"-I{i}" for i in inc] + ["-o", str(exe), str(src)], check=True)
    out = subprocess.run([str(exe)], capture_output=True, text=True, env={**os.environ, "CUDA_VISIBLE_DEVICES": ""})
    assert out.returncode == 0, out.stdout
