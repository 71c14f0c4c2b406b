"""Kernels and dispatch branches at the sizes where they can go wrong, against the CPU oracle."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_2209_13443_b200 import workloads as wl
from tests import util

pytestmark = pytest.mark.gpu


# fp32 convolutions: H, W, cin, cout, k, stride, pad, residual
F32_GEOMS = [
    (9, 6, 12, 40, 3, 1, 1, True),       # K < 128: one K group, ragged M and N
    (57, 55, 16, 72, 3, 1, 1, True),     # 64 x 64 tiles, two K groups, K tail inside a ring stage
    (8, 8, 136, 72, 3, 1, 1, False),     # 32 x 32 tiles, a cluster cuts K
    (2, 1, 512, 64, 3, 1, 1, True),      # 16 x 32 tiles, K = 4608 over eight CTAs
    (3, 1, 150, 33, 3, 1, 1, False),     # 4-byte copies (Cin not a multiple of 4), last CTA's K range short, odd N
    (6, 5, 37, 8, 2, 1, 0, False),       # K = 148: one full ring stage and a tail
]


@pytest.mark.parametrize("geom", F32_GEOMS)
def test_fp32_convolution_tiles_and_k_cuts(geom):
    H, W, cin, cout, k, stride, pad, residual = geom
    spec = util.single_layer_model("f32", H, W, cin, cout, k, stride, pad, wl.ACT_RELU, residual, seed=sum(geom), max_batch=5)
    run = util.GpuRunner(spec)
    alone = {}
    for B in (1, 5):
        x = wl.random_features((5, H, W, cin), seed=2, bf16=False, relu=False)[:B]
        g = run.stage(0, x)
        util.check_stage(spec, g, util.oracle_stage(spec, 0, x), f"f32 {geom} B={B}", elementwise=True)
        alone[B] = g["features_out"][0]
    assert np.array_equal(alone[1], alone[5])     # the cut of K does not depend on the batch
