"""Kernels and dispatch branches at the sizes where they can go wrong, against the CPU oracle."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from oracle import ee_oracle as eo
from paper_2209_13443_b200 import binding as eb
from paper_2209_13443_b200 import workloads as wl
from tests import util

pytestmark = pytest.mark.gpu


# fp32 convolutions: H, W, cin, cout, k, stride, pad, residual
F32_GEOMS = [
    (9, 6, 12, 40, 3, 1, 1, True),       # K < 128: one K group, ragged M and N
    (57, 55, 16, 72, 3, 1, 1, True),     # 64 x 64 tiles, two K groups, K tail inside a ring stage
    (8, 8, 136, 72, 3, 1, 1, False),     # 32 x 32 tiles, a cluster cuts K
    (2, 1, 512, 64, 3, 1, 1, True),      # 16 x 32 tiles, K = 4608 over eight CTAs
    (2, 3, 136, 40, 3, 1, 1, True),      # 30 rows at the largest batch: two of them
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


# exit heads: dtype, B, HW, C, K: every tile height and cluster size, channels that leave a ring slot ragged, class blocks
# that are short or empty, classes past one block per CTA, C the cluster kernel does not take
HEADS = [("bf16", 3, 4, 520, 1000), ("bf16", 13, 9, 8, 17), ("bf16", 64, 2, 2048, 1000), ("bf16", 17, 3, 264, 129), ("bf16", 5, 5, 256, 5000),
         ("bf16", 7, 6, 20, 33), ("f32", 1, 4, 132, 70), ("f32", 33, 2, 64, 10), ("f32", 6, 4, 2048, 100), ("f32", 9, 3, 7, 12)]


@pytest.mark.parametrize("case", HEADS)
def test_fc_cluster_tiles_against_the_oracle_and_alone(case):
    dtype, B, HW, C, K = case
    bf16 = dtype == "bf16"
    rng = wl._rng(B + C + K, 907)
    fw, fb = wl._head(rng, C, K, 4.0, bf16)
    layers = [wl._conv(rng, wl.OP_CONV, C, C, 1, 1, 0, wl.ACT_NONE, bf16=bf16)]
    spec = wl.Model("head", dtype, 1, HW, C, [wl.Stage(layers, K, fw, fb, 0.5, False)], B)
    m = eb.EEModel(spec)
    out = eb.StageBuffers(m, 0)
    scratch = torch.empty(m.exit_head_scratch_bytes(0) + 256, dtype=torch.uint8, device="cuda")
    x = wl.random_features((B, HW, C), seed=3, bf16=bf16)
    shift = (np.arange(B) % 3 == 0).astype(np.float32) * 12.0
    cls = (np.arange(B) * 7 % K).astype(np.int32)
    xd, sd, cd = eb.to_device(dtype, x), torch.as_tensor(shift, device="cuda"), torch.as_tensor(cls, device="cuda")
    for _ in range(2):      # the second call: the counters of the first are back at zero
        m.exit_head(0, xd, B, HW, out, scratch, sd, cd)
    torch.cuda.synchronize()
    z, conf, mask = out.logits[:B].cpu().numpy(), out.conf[:B].cpu().numpy(), out.exit_mask[:B].cpu().numpy()
    o = eo.exit_head(x, fw, fb, 0.5, False, shift, cls)
    assert util.rel_err(z, o["z"], dtype, floor=util.LOGIT_FLOOR[dtype]) <= util.TOL[dtype]
    assert np.max(np.abs(conf - o["conf"])) <= util.TOL[dtype]
    sure = np.abs(o["conf"] - 0.5) > util.BAND
    assert np.array_equal(mask[sure], o["exit"][sure])
    n = int(out.n_surv_dev[0])
    assert np.array_equal(out.survivor_idx[:n].cpu().numpy(), np.nonzero(mask == 0)[0]) and n == B - int(mask.sum())
    b = B - 1               # alone: another tile height and cluster size, the same bits
    m.exit_head(0, xd[b:].contiguous(), 1, HW, out, scratch, sd[b:].contiguous(), cd[b:].contiguous())
    torch.cuda.synchronize()
    assert np.array_equal(out.logits[0].cpu().numpy(), z[b]) and float(out.conf[0]) == float(conf[b])


def test_stage_replay_on_the_default_stream_is_bit_identical():
    spec = wl.resnet50_ee(seed=1, in_hw=64, n_classes=100, max_batch=6)
    run = util.GpuRunner(spec)
    xd = eb.to_device("bf16", wl.make_input(spec, 5, seed=3))
    out, snaps = run.bufs[0], []
    default = torch.cuda.default_stream()
    for graphs in (False, True, True):
        run.m.set_graphs(graphs)
        out.logits.fill_(0)
        torch.cuda.synchronize()
        out.arm_count()
        run.m.stage_run(0, xd, 5, out, run.ws, stream=default)
        n = out.wait_count()
        torch.cuda.synchronize()
        snaps.append((n, out.logits[:5].clone(), out.features_out[:n].clone()))
    for n, z, f in snaps[1:]:
        assert n == snaps[0][0] == int(out.n_surv_dev[0]) and torch.equal(z, snaps[0][1]) and torch.equal(f, snaps[0][2])


def test_stage_outputs_of_a_new_buffer_set_are_not_those_of_a_dead_one():
    """run_until_exit keeps the ee_stage_out_t array of the last buffer set; a new set may have the ids of a dead one."""
    spec = wl.tiny_ee_cnn(seed=0)
    m = eb.EEModel(spec)
    ws = m.workspace()
    x = eb.to_device("f32", wl.make_input(spec, 4, seed=1))
    for _ in range(4):
        bufs = [eb.StageBuffers(m, s) for s in range(m.n_stages)]
        bufs[0].conf.fill_(-1.0)
        m.run_until_exit(0, x, 4, bufs, ws)
        torch.cuda.synchronize()
        assert bool((bufs[0].conf[:4] > 0).all())
        del bufs


# convolutions with several taps: H, W, cin, cout, kh, kw, stride, pad, pad_w, max_batch
TAP_GEOMS = [
    (14, 14, 128, 256, 3, 3, 1, 1, 1, 5),     # whole channel blocks, ragged last tile
    (7, 7, 192, 96, 3, 3, 1, 1, 1, 5),        # a tile over three images, 96 filters
    (28, 28, 72, 128, 3, 3, 2, 1, 1, 3),      # stride 2: even rows first, then odd ones; ragged channel block
    (9, 13, 64, 40, 3, 3, 2, 1, 1, 3),        # the same, odd sizes, fewer than 64 filters
    (17, 17, 96, 96, 1, 7, 1, 0, 3, 2),       # one filter row
    (17, 17, 96, 96, 7, 1, 1, 3, 0, 2),       # one filter column
    (6, 70, 64, 16, 3, 3, 1, 1, 1, 2),        # rows wider than half a tile, 16 filters
    (3, 128, 16, 24, 5, 3, 1, 2, 1, 1),       # 24 filters, five filter rows
    (1, 1, 64, 200, 3, 3, 1, 1, 1, 9),        # one pixel per image
    (11, 11, 64, 72, 5, 5, 2, 2, 2, 4),       # stride 2, three even and two odd rows
]


@pytest.mark.parametrize("geom", TAP_GEOMS)
def test_convolution_with_several_taps(geom):
    H, W, cin, cout, kh, kw, stride, pad, pad_w, bmax = geom
    rng = wl._rng(sum(geom), 911)
    layer = wl._conv_hw(rng, cin, cout, kh, kw, stride, pad, pad_w, wl.ACT_RELU, bf16=True)
    fw, fb = wl._head(rng, cout, 7, 1.0, True)
    spec = wl.Model("taps", "bf16", H, W, cin, [wl.Stage([layer], 7, fw, fb, 2.0, False)], bmax)
    run = util.GpuRunner(spec)
    first = {}
    for B in sorted({1, bmax}):
        x = wl.random_features((bmax, H, W, cin), seed=4, bf16=True, relu=False)[:B]
        g = run.stage(0, x)
        util.check_stage(spec, g, util.oracle_stage(spec, 0, x), f"{geom} B={B}", elementwise=True)
        first[B] = g["features_out"][0]
    # the sums do not depend on the batch
    assert np.array_equal(first[1], first[bmax])


# one-wave tiles: H, W, cin, cout, k, stride, residual, batches (32-, 64-, 128-filter tiles, then CTAs that share SMs): one K block,
# as many as slots and one more, ragged pixels, filters and channels, a tile over several images
WAVE_GEOMS = [
    (14, 14, 64, 256, 1, 1, True, (1, 13, 24, 49)), (7, 7, 704, 136, 1, 1, True, (2, 65)), (7, 7, 768, 512, 1, 1, False, (1, 24, 50, 97)),
    (9, 11, 200, 40, 3, 1, False, (1, 5)), (13, 13, 72, 264, 3, 2, True, (3, 40, 90)), (8, 8, 128, 8, 3, 1, True, (1, 7)),
]


@pytest.mark.parametrize("geom", WAVE_GEOMS)
def test_one_wave_tiles_against_the_oracle_and_at_every_width(geom):
    H, W, cin, cout, k, stride, residual, batches = geom
    spec = util.single_layer_model("bf16", H, W, cin, cout, k, stride, k // 2, wl.ACT_RELU, residual, seed=sum(geom[:6]), max_batch=batches[-1])
    run = util.GpuRunner(spec)
    for i in range(len(spec.stages[0].layers)):
        run.m.set_layer_splits(0, i, 1)
    first = None
    for B in batches:
        x = wl.random_features((batches[-1], H, W, cin), seed=6, bf16=True, relu=False)[:B]
        g = run.stage(0, x)
        if first is None:
            util.check_stage(spec, g, util.oracle_stage(spec, 0, x), f"{geom} B={B}", elementwise=not residual)
            first = g["features_out"]
        assert np.array_equal(g["features_out"][: len(first)], first), f"{geom} B={B}"


# one-wave tiles of 64 pixels (32 and 64 filters) and of 128 x 32: K blocks that leave a group short, exactly as many as the ring has
# slots and one more, a ragged last tile, images that straddle tiles
WAVE_GROUP_GEOMS = [
    (8, 8, 1024, 512, 1, 1, False, (1, 9, 10, 18, 19)), (8, 8, 1088, 520, 1, 1, True, (1, 8, 17)), (14, 14, 704, 96, 1, 1, True, (1, 23, 25, 32)),
    (7, 7, 192, 512, 3, 1, True, (1, 3, 12)), (5, 5, 320, 72, 1, 1, False, (1, 2, 60)), (7, 7, 832, 256, 1, 1, False, (1, 40)),
]


@pytest.mark.parametrize("geom", WAVE_GROUP_GEOMS)
def test_one_wave_tiles_of_64_pixels_and_groups_of_k_blocks(geom):
    test_one_wave_tiles_against_the_oracle_and_at_every_width(geom)


@pytest.mark.parametrize("case", [(7, 7, 64, 40, 128, 1, 1), (14, 14, 128, 520, 96, 2, 2), (5, 9, 320, 256, 704, 1, 3), (14, 14, 64, 1000, 72, 1, 5), (14, 14, 192, 1016, 136, 1, 9)])
def test_projection_inside_a_one_wave_tile_gives_the_bits_of_two_layers(case):
    H, W, mid, wide, cin, stride, B = case
    rng = wl._rng(H + wide, 917)
    conv = lambda ci, co, s, act, src, res=wl.NO_RESIDUAL: wl._conv(rng, wl.OP_CONV, ci, co, 1, s, 0, act, bf16=True, input_from=src, residual_from=res)  # noqa: E731
    layers = [conv(cin, mid, stride, wl.ACT_RELU, wl.FROM_STAGE_INPUT), conv(cin, wide, stride, wl.ACT_NONE, wl.FROM_STAGE_INPUT),
              conv(mid, wide, 1, wl.ACT_RELU, 0, 1)]
    fw, fb = wl._head(rng, wide, 5, 1.0, True)
    spec = wl.Model("proj", "bf16", H, W, cin, [wl.Stage(layers, 5, fw, fb, 2.0, False)], B)
    run = util.GpuRunner(spec)
    x = eb.to_device("bf16", wl.random_features((B, H, W, cin), seed=8, bf16=True))
    got = []
    for fused in (True, False):
        run.m.set_proj_fusion(fused)
        run.bufs[0].features_out.fill_(0)
        run.m.stage_run(0, x, B, run.bufs[0], run.ws)
        torch.cuda.synchronize()
        run.m.check()
        got.append(run.bufs[0].features_out[:B].clone())
        assert sum(p["launches"] for p in run.m.plan(0, B)) == (2 if fused else 3)
    assert torch.equal(*got) and bool(got[0].any())


# stems: H, W, cout, k, activation, B: rows of an odd number of elements (the batch's last one alone in its word), 128 output columns,
# one output row, ranges that start inside an image, one and two channel halves
STEMS = [(161, 161, 64, 7, wl.ACT_RELU, 3), (15, 33, 8, 7, wl.ACT_NONE, 1), (9, 255, 40, 7, wl.ACT_RELU6, 2), (1, 5, 64, 7, wl.ACT_NONE, 3),
         (63, 65, 32, 3, wl.ACT_RELU6, 5), (20, 256, 64, 3, wl.ACT_RELU, 2), (2, 1, 48, 3, wl.ACT_NONE, 2)]


@pytest.mark.parametrize("case", STEMS)
def test_stem_kernels_with_and_without_the_pool(case):
    H, W, cout, k, act, B = case
    rng = wl._rng(H + W, 919)
    layers = [wl._conv(rng, wl.OP_CONV, 3, cout, k, 2, k // 2, act, bf16=True), wl.Layer(wl.OP_MAXPOOL, cout, cout, 3, 3, 2, 1)]
    fw, fb = wl._head(rng, cout, 5, 1.0, True)
    spec = wl.Model("stem", "bf16", H, W, 3, [wl.Stage(layers, 5, fw, fb, 2.0, False)], B)
    run = util.GpuRunner(spec)
    m, out = run.m, run.bufs[0]
    assert [pl["launches"] for pl in m.plan(0, B)] == [1, 0]
    x = wl.make_input(spec, B, seed=5)
    xd = eb.to_device("bf16", x)
    shapes = wl.stage_shapes(spec)[0]["layers"]
    conv, apart = (torch.empty((B,) + s, dtype=torch.bfloat16, device="cuda") for s in shapes)
    m.layer_run(0, 0, xd, None, B, conv, run.ws)
    m.layer_run(0, 1, conv, None, B, apart, run.ws)
    m.stage_run(0, xd, B, out, run.ws)
    torch.cuda.synchronize()
    m.check()
    assert torch.equal(out.features_out[:B], apart)
    assert util.rel_err(apart.float().cpu().numpy(), eo.run_layers(spec, 0, x), "bf16") <= util.TOL["bf16"]
    m.stage_run(0, xd[B - 1:].clone(), 1, out, run.ws)      # alone: other row ranges, the same bits
    torch.cuda.synchronize()
    assert torch.equal(out.features_out[0], apart[B - 1])
    run.check_guards()


@pytest.mark.parametrize("fused", [False, True])
def test_decisions_in_pinned_memory_are_there_when_the_count_is(fused):
    spec = wl.resnet50_ee(seed=1, in_hw=64, n_classes=100, max_batch=64)
    m = eb.EEModel(spec)
    m.set_fused_head(fused)
    ws = m.workspace()
    dev, pin = eb.StageBuffers(m, 0), eb.StageBuffers(m, 0, pinned_decisions=True)
    for B in (1, 17, 64):
        x = eb.to_device("bf16", wl.make_input(spec, B, seed=B))
        m.stage_run(0, x, B, dev, ws)
        torch.cuda.synchronize()
        for _ in range(3):
            pin.conf.fill_(-1)
            pin.pred.fill_(-1)
            pin.arm_count()
            m.stage_run(0, x, B, pin, ws)
            n = pin.wait_count()
            assert n == int(dev.n_surv_dev[0]) and torch.equal(pin.conf[:B], dev.conf[:B].cpu()) and torch.equal(pin.pred[:B], dev.pred[:B].cpu())


# 3x3 layers on 64 channels: H, W, cout, B: one and two channel halves, a half of one vector, one image row per tile, ragged last bands
@pytest.mark.parametrize("geom", [(56, 56, 64, 3), (13, 61, 8, 2), (5, 20, 40, 4), (1, 1, 32, 2), (17, 30, 48, 3)])
def test_halo_epilogue_of_narrow_and_wide_layers(geom):
    H, W, cout, B = geom
    spec = util.single_layer_model("bf16", H, W, 64, cout, 3, 1, 1, wl.ACT_RELU6, False, seed=sum(geom), max_batch=B)
    run = util.GpuRunner(spec)
    x = wl.random_features((B, H, W, 64), seed=9, bf16=True, relu=False)
    util.check_stage(spec, run.stage(0, x), util.oracle_stage(spec, 0, x), f"{geom}", elementwise=True)
    run.check_guards()


# heads on more channels or classes than a tile of eight samples has shared memory for: tiles of four, two and one, the last channel
# count the cluster kernel takes and one that it does not
WIDE_HEADS = [("bf16", 64, 3072, 1000), ("bf16", 19, 8192, 40), ("bf16", 9, 24064, 12), ("bf16", 9, 24576, 12), ("bf16", 33, 64, 30000), ("f32", 37, 8192, 300), ("f32", 5, 16384, 7)]


@pytest.mark.parametrize("case", WIDE_HEADS)
def test_wide_heads_against_the_oracle_and_alone(case):
    dtype, B, C, K = case
    bf16 = dtype == "bf16"
    rng = wl._rng(B + C + K, 911)
    fw, fb = wl._head(rng, C, K, 4.0, bf16)
    spec = wl.Model("wide head", dtype, 1, 2, C, [wl.Stage([wl.Layer(wl.OP_MAXPOOL, C, C, 3, 3, 1, 1)], K, fw, fb, 0.5, False)], B)
    m = eb.EEModel(spec)
    out = eb.StageBuffers(m, 0)
    scratch, guard = util.guarded((m.exit_head_scratch_bytes(0) + 256,), torch.uint8)
    x = wl.random_features((B, 2, C), seed=3, bf16=bf16)
    xd = eb.to_device(dtype, x)
    for _ in range(2):
        m.exit_head(0, xd, B, 2, out, scratch)
    torch.cuda.synchronize()
    m.check()
    z, conf, mask = out.logits[:B].cpu().numpy(), out.conf[:B].cpu().numpy(), out.exit_mask[:B].cpu().numpy()
    o = eo.exit_head(x, fw, fb, 0.5, False, None, None)
    assert util.rel_err(z, o["z"], dtype, floor=util.LOGIT_FLOOR[dtype]) <= util.TOL[dtype]
    assert np.max(np.abs(conf - o["conf"])) <= util.TOL[dtype]
    n = int(out.n_surv_dev[0])
    assert np.array_equal(out.survivor_idx[:n].cpu().numpy(), np.nonzero(mask == 0)[0]) and n == B - int(mask.sum())
    assert bool(torch.all(guard == util.CANARY))
    b = B - 1
    m.exit_head(0, xd[b:].contiguous(), 1, 2, out, scratch)
    torch.cuda.synchronize()
    assert np.array_equal(out.logits[0].cpu().numpy(), z[b]) and float(out.conf[0]) == float(conf[b])


# 3x3 512->512 (72 K blocks): whole where the largest batch would not run as deep clusters, four K ranges where it does
@pytest.mark.parametrize("hw,bmax,ranges", [(6, 64, 1), (4, 64, 1), (6, 16, 4), (2, 64, 4)])
def test_k_ranges_chosen_for_a_layer_and_its_results(hw, bmax, ranges):
    spec = util.single_layer_model("bf16", hw, hw, 512, 512, 3, 1, 1, wl.ACT_RELU, False, seed=hw, max_batch=bmax)
    run = util.GpuRunner(spec)
    assert run.m.layer_config(0, 0, 1)["splits"] == ranges
    x = wl.random_features((bmax, hw, hw, 512), seed=3, bf16=True, relu=False)
    whole = run.stage(0, x)
    # the layer's output: the logits of such small maps are sums of a few rounded values that cancel, not the layer's to bound
    assert util.rel_err(whole["features_out"], eo.run_layers(spec, 0, x), "bf16") <= util.TOL["bf16"]
    assert np.array_equal(run.stage(0, x[:1])["features_out"][0], whole["features_out"][0])


# K ranges on the one-wave kernel, every tile that takes them (64 x 32, 64 x 64, 128 x 32, 128 x 64): the bits of a cluster of CTAs per
# tile; a last range that is shorter, ranges that end inside a group of K blocks, ragged filters: H, W, cin, cout, residual, ranges, batches
WAVE_RANGE_GEOMS = [(7, 7, 512, 512, False, 4, (1, 12, 40)), (14, 14, 200, 96, True, 3, (1, 20, 30, 40)), (9, 9, 136, 64, False, 5, (1, 7)),
                    (5, 5, 320, 72, True, 2, (1, 3, 40))]


@pytest.mark.parametrize("geom", WAVE_RANGE_GEOMS)
def test_k_ranges_on_the_one_wave_kernel_give_the_bits_of_the_cluster(geom):
    H, W, cin, cout, residual, ranges, batches = geom
    spec = util.single_layer_model("bf16", H, W, cin, cout, 3, 1, 1, wl.ACT_RELU, residual, seed=cin, max_batch=batches[-1])
    layer = 1 if residual else 0
    m = eb.EEModel(spec)
    m.set_layer_splits(0, layer, ranges)
    ws = m.workspace()
    for B in batches:
        xd = eb.to_device("bf16", wl.random_features((B, H, W, cin), seed=B, bf16=True, relu=False))
        res = eb.to_device("bf16", wl.random_features((B, H, W, cout), seed=B + 1, bf16=True)) if residual else None
        got = {}
        for variant in (0, 3):
            m.set_layer_variant(0, layer, 1, batches[-1], variant)
            got[variant], guard = util.guarded((B, H, W, cout), torch.bfloat16)
            m.layer_run(0, layer, xd, res, B, got[variant], ws)
            torch.cuda.synchronize()
            m.check()
            assert bool(torch.all(guard == util.CANARY))
        assert torch.equal(got[0], got[3])


# NaN and infinities through the pooling stem: the pooling layer run apart drops NaN, and a window of nothing else is -inf
@pytest.mark.parametrize("act", [wl.ACT_RELU, wl.ACT_RELU6, wl.ACT_NONE])
@pytest.mark.parametrize("k,cout", [(7, 64), (3, 40)])
def test_pooling_stem_treats_nan_as_the_two_layers_run_apart(k, cout, act):
    H, W, B = 37, 61, 2
    rng = wl._rng(k + act, 921)
    layers = [wl._conv(rng, wl.OP_CONV, 3, cout, k, 2, k // 2, act, bf16=True), wl.Layer(wl.OP_MAXPOOL, cout, cout, 3, 3, 2, 1)]
    fw, fb = wl._head(rng, cout, 5, 1.0, True)
    spec = wl.Model("stem", "bf16", H, W, 3, [wl.Stage(layers, 5, fw, fb, 2.0, False)], B)
    m = eb.EEModel(spec)
    out, ws = eb.StageBuffers(m, 0), m.workspace()
    xd = eb.to_device("bf16", wl.make_input(spec, B, seed=5))
    xd[0, 4:30, 6:33] = float("nan")                 # whole windows of NaN
    xd[1, ::17, ::13, 1] = float("nan")
    xd[1, 5, 5, 0], xd[1, 20, 30, 2], xd[0, 35, 2] = float("inf"), float("-inf"), float("inf")
    shapes = wl.stage_shapes(spec)[0]["layers"]
    conv, apart = (torch.empty((B,) + s, dtype=torch.bfloat16, device="cuda") for s in shapes)
    m.layer_run(0, 0, xd, None, B, conv, ws)
    m.layer_run(0, 1, conv, None, B, apart, ws)
    m.stage_run(0, xd, B, out, ws)
    torch.cuda.synchronize()
    m.check()
    if act != wl.ACT_RELU6:                          # min(max(x, 0), 6) has no NaN
        assert bool(conv.isnan().any()) and bool((apart == float("-inf")).any())
    assert not bool(apart.isnan().any())
    assert torch.equal(out.features_out[:B].view(torch.int16), apart.view(torch.int16))


# survivors close up in place, or are gathered where features_out is not 16-byte aligned: dtype, HW, C (rows of 16-, 2- and 4-byte units)
@pytest.mark.parametrize("dtype,hw,c", [("bf16", 7, 64), ("bf16", 3, 9), ("f32", 5, 12), ("f32", 3, 5), ("bf16", 3, 10)])
@pytest.mark.parametrize("aligned", [True, False])
def test_survivors_close_up_in_place(dtype, hw, c, aligned):
    B = 40
    spec = util.single_layer_model(dtype, hw, hw, c, c, 1, 1, 0, wl.ACT_RELU, False, seed=c, max_batch=B)
    s0 = spec.stages[0]
    s0.threshold, s0.fc_weight = 0.9, s0.fc_weight * 0.0
    m = eb.EEModel(spec)
    ws, out = m.workspace(), eb.StageBuffers(m, 0)
    n_el = out.features_out.numel()
    flat, guard = util.guarded((n_el + 8,), out.features_out.dtype)
    off = 0 if aligned else 1
    out.features_out = flat[off:off + n_el].view(out.features_out.shape)
    x = eb.to_device(dtype, wl.random_features((B, hw, hw, c), seed=3, bf16=dtype == "bf16"))
    full = torch.empty((B, hw, hw, c), dtype=x.dtype, device="cuda")
    m.layer_run(0, 0, x, None, B, full, ws)
    rng = np.random.default_rng(5)
    masks = [np.zeros(B, bool), np.ones(B, bool), np.arange(B) == 0, np.arange(B) == B - 1, np.arange(B) == 17, np.arange(B) % 2 == 0,
             np.arange(B) < 39, np.arange(B) >= 16, rng.random(B) < 0.3, rng.random(B) < 0.7]
    for leave in masks:
        for b in (B, 16, 1):
            lv = leave[:b]
            shift = torch.as_tensor(lv.astype(np.float32) * 30.0, device="cuda")
            m.stage_run(0, x, b, out, ws, None, shift, torch.zeros(b, dtype=torch.int32, device="cuda"))
            torch.cuda.synchronize()
            stay = np.nonzero(~lv)[0]
            n = int(out.n_surv_dev[0])
            assert n == len(stay) and np.array_equal(out.survivor_idx[:n].cpu().numpy(), stay)
            assert torch.equal(out.features_out[:n], full[torch.as_tensor(stay, device="cuda")])
    m.check()
    assert bool(torch.all(guard == util.CANARY))


# the FC kernel pools by itself (one pass of its threads over a map), one pass more than that, warps that share a class's channels, and
# 56 samples, whose survivors are one word, and 57, which scan: dtype, B, max_batch, HW, C, K
HEAD_ROUTES = [("f32", 8, 8, 256, 64, 10), ("f32", 8, 8, 256, 68, 10), ("bf16", 5, 6, 784, 64, 33), ("bf16", 3, 6, 784, 72, 64), ("f32", 3, 6, 8, 520, 100),
               ("f32", 6, 32, 4, 2048, 17), ("bf16", 13, 32, 5, 1032, 129), ("bf16", 56, 64, 3, 40, 1000), ("bf16", 57, 64, 3, 40, 1000), ("f32", 56, 57, 16, 16, 10),
               ("f32", 57, 57, 16, 16, 10), ("bf16", 1, 1, 49, 16, 10)]


POOLED = [(256, 64, 10), (784, 64, 33), (16, 16, 10), (49, 16, 10)]


@pytest.mark.parametrize("case", HEAD_ROUTES)
def test_head_routes_against_the_oracle_and_alone(case):
    dtype, B, most, HW, C, K = case
    bf16 = dtype == "bf16"
    rng = wl._rng(B + C + K, 923)
    fw, fb = wl._head(rng, C, K, 4.0, bf16)
    spec = wl.Model("routes", dtype, 1, HW, C, [wl.Stage([wl.Layer(wl.OP_MAXPOOL, C, C, 3, 3, 1, 1)], K, fw, fb, 0.5, False)], most)
    m = eb.EEModel(spec)
    assert m.head_pools(0, B) == int((HW, C, K) in POOLED)
    out, pin = eb.StageBuffers(m, 0), eb.StageBuffers(m, 0, pinned_decisions=True)
    scratch, guard = util.guarded((m.exit_head_scratch_bytes(0) + 256,), torch.uint8)
    scratch.fill_(0x5A)
    x = wl.random_features((B, HW, C), seed=3, bf16=bf16)
    xd = eb.to_device(dtype, x)
    shift, cls = (np.arange(B) % 3 == 0).astype(np.float32) * 12.0, (np.arange(B) * 7 % K).astype(np.int32)
    sd, cd = torch.as_tensor(shift, device="cuda"), torch.as_tensor(cls, device="cuda")
    for o in (out, pin, out):      # the counters of a call are back at zero for the next
        m.exit_head(0, xd, B, HW, o, scratch, sd, cd)
    torch.cuda.synchronize()
    m.check()
    z, conf, mask = out.logits[:B].cpu().numpy(), out.conf[:B].cpu().numpy(), out.exit_mask[:B].cpu().numpy()
    o = eo.exit_head(x, fw, fb, 0.5, False, shift, cls)
    assert util.rel_err(z, o["z"], dtype, floor=util.LOGIT_FLOOR[dtype]) <= util.TOL[dtype]
    sure = np.abs(o["conf"] - 0.5) > util.BAND
    assert np.array_equal(mask[sure], o["exit"][sure])
    n = int(out.n_surv_dev[0])
    assert np.array_equal(out.survivor_idx[:n].cpu().numpy(), np.nonzero(mask == 0)[0]) and n == B - int(mask.sum())
    assert torch.equal(pin.conf[:B], out.conf[:B].cpu()) and bool(torch.all(guard == util.CANARY))
    m.exit_head(0, xd[B - 1:].contiguous(), 1, HW, out, scratch, sd[B - 1:].contiguous(), cd[B - 1:].contiguous())
    torch.cuda.synchronize()
    assert np.array_equal(out.logits[0].cpu().numpy(), z[B - 1]) and float(out.conf[0]) == float(conf[B - 1])


# heads whose tiles are clusters: 16 CTAs a tile, survivors in one word; two CTAs and the scan of more than 56 samples; eight CTAs whose warps share classes
@pytest.mark.parametrize("case", [("bf16", 5, 64, 9, 64, 1000), ("bf16", 37, 64, 9, 64, 1000), ("f32", 60, 64, 16, 16, 100), ("f32", 6, 32, 4, 2048, 100)])
def test_head_whose_exchange_runs_out_of_time_is_reported_and_keeps_its_samples(case):
    """With a limit of one clock the wait for the tile's triples runs out.  The call ends all the same, the time-out is reported once, and a sample whose
    triples were late stays in the batch, with confidence 0; one whose triples were there is decided as ever."""
    dtype, B, most, HW, C, K = case
    fw, fb = wl._head(wl._rng(B + C + K, 924), C, K, 4.0, dtype == "bf16")
    spec = wl.Model("late", dtype, 1, HW, C, [wl.Stage([wl.Layer(wl.OP_MAXPOOL, C, C, 3, 3, 1, 1)], K, fw, fb, 0.5, False)], most)
    m = eb.EEModel(spec)
    scratch = torch.empty(m.exit_head_scratch_bytes(0) + 256, dtype=torch.uint8, device="cuda")
    x = eb.to_device(dtype, wl.random_features((B, HW, C), seed=3, bf16=dtype == "bf16"))
    shift = torch.as_tensor((np.arange(B) % 3 == 0).astype(np.float32) * 40.0, device="cuda")   # these leave
    cls = torch.as_tensor((np.arange(B) * 7 % K).astype(np.int32), device="cuda")
    right, late, again = (eb.StageBuffers(m, 0) for _ in range(3))

    def call(out):
        m.exit_head(0, x, B, HW, out, scratch, shift, cls)
        torch.cuda.synchronize()
        return out.conf[:B].cpu().numpy(), out.pred[:B].cpu().numpy(), out.exit_mask[:B].cpu().numpy(), out.logits[:B].cpu().numpy()

    want = call(right)
    m.check()
    assert want[2][::3].all()
    m.set_wait_limit(1)
    for _ in range(20):   # a leader that happens to be its cluster's last has nothing to wait for
        conf, pred, mask, z = call(late)
        gone = conf == 0.0
        if gone.any():
            break
    with pytest.raises(eb.EEError) as e:
        m.check()
    assert e.value.status == 7                                         # EE_ERR_TIMEOUT
    assert gone.any() and not pred[gone].any() and not mask[gone].any()
    for got, w in zip((conf, pred, mask), want):
        assert np.array_equal(got[~gone], w[~gone])
    assert np.array_equal(z, want[3])
    n = int(late.n_surv_dev[0])
    assert n == B - int(mask.sum()) and np.array_equal(late.survivor_idx[:n].cpu().numpy(), np.nonzero(mask == 0)[0])
    m.set_wait_limit(4_000_000_000)
    for got, w in zip(call(again), want):
        assert np.array_equal(got, w)
    m.check()


# rows of a map, its blocks of G rows and row groups: one row a block with two, three and more than eight blocks a group, two rows likewise; 16 and 32
# rows, whose blocks two lanes share at few samples: fewer blocks than groups, as many, one more
@pytest.mark.parametrize("HW,G,groups", [(63, 1, 32), (65, 1, 64), (127, 1, 64), (129, 1, 64), (513, 1, 64), (1681, 1, 64), (258, 2, 64), (1026, 2, 64), (98, 2, 32),
                                         (48, 16, 8), (784, 16, 32), (1040, 16, 64), (96, 32, 8), (1056, 32, 32), (2048, 32, 64), (3136, 32, 64)])
def test_pooling_adds_the_blocks_of_a_row_group_in_order(HW, G, groups):
    B, C = 2, 72
    spec = wl.Model("rows", "bf16", 1, HW, C, [wl.Stage([wl.Layer(wl.OP_MAXPOOL, C, C, 3, 3, 1, 1)], C, np.eye(C, dtype=np.float32), None, 0.5, False)], B)
    m = eb.EEModel(spec)
    out = eb.StageBuffers(m, 0)
    scratch = torch.empty(m.exit_head_scratch_bytes(0) + 256, dtype=torch.uint8, device="cuda")
    x = wl.random_features((B, HW, C), seed=HW, bf16=True, relu=False)
    m.exit_head(0, eb.to_device("bf16", x), B, HW, out, scratch)
    torch.cuda.synchronize()
    blocks = np.asarray(x, dtype=np.float32).reshape(B, HW // G, G, C)
    while blocks.shape[2] > 1:      # the pairwise tree over a block's rows
        blocks = blocks[:, :, :blocks.shape[2] // 2] + blocks[:, :, blocks.shape[2] // 2:]
    blocks, want = blocks[:, :, 0], np.zeros((B, C), dtype=np.float32)
    for q in range(groups):
        part = np.zeros((B, C), dtype=np.float32)
        for j in range(q, HW // G, groups):
            part = part + blocks[:, j]
        want = want + part
    assert np.array_equal(out.logits[:B].cpu().numpy(), want / np.float32(HW))   # the FC layer is the identity: the logits are the pooled vector


# 16- and 32-row blocks at batches on both sides of the line up to which two lanes share them (a quarter of 148 SMs, in CTAs): rows, G, groups, channels, most samples
@pytest.mark.parametrize("HW,G,groups,C,most", [(48, 16, 8, 72, 41), (784, 16, 32, 72, 41), (1040, 16, 64, 72, 41), (96, 32, 8, 72, 41), (1056, 32, 32, 72, 41), (3136, 32, 64, 72, 41),
                                                (784, 16, 32, 512, 12), (3136, 32, 64, 256, 12)])
def test_pooled_sums_do_not_depend_on_the_batch(HW, G, groups, C, most):
    spec = wl.Model("rows", "bf16", 1, HW, C, [wl.Stage([wl.Layer(wl.OP_MAXPOOL, C, C, 3, 3, 1, 1)], C, np.eye(C, dtype=np.float32), None, 0.5, False)], most)
    m = eb.EEModel(spec)
    out = eb.StageBuffers(m, 0)
    scratch = torch.empty(m.exit_head_scratch_bytes(0) + 256, dtype=torch.uint8, device="cuda")
    x = wl.random_features((most, HW, C), seed=HW, bf16=True, relu=False)
    xd = eb.to_device("bf16", x)
    blocks = np.asarray(x, dtype=np.float32).reshape(most, HW // G, G, C)
    while blocks.shape[2] > 1:      # the pairwise tree over a block's rows
        blocks = blocks[:, :, :blocks.shape[2] // 2] + blocks[:, :, blocks.shape[2] // 2:]
    blocks, want = blocks[:, :, 0], np.zeros((most, C), dtype=np.float32)
    for q in range(groups):
        part = np.zeros((most, C), dtype=np.float32)
        for j in range(q, HW // G, groups):
            part = part + blocks[:, j]
        want = want + part
    for B in (most, 13, 12, 1):
        if B > most:
            continue
        m.exit_head(0, xd, B, HW, out, scratch)
        torch.cuda.synchronize()
        assert np.array_equal(out.logits[:B].cpu().numpy(), want[:B] / np.float32(HW)), B   # the FC layer is the identity


# 1x1 layer + depthwise layer in one launch: H, W, cin, hidden, stride, batches: one to three K blocks, channel blocks that are short, odd
# or not a multiple of 16, bands of one row and of the whole image, one pixel, the widest row, images smaller than a tile of positions
XDW_GEOMS = [(14, 14, 64, 384, 1, (1, 5)), (7, 7, 160, 960, 1, (1, 9)), (20, 50, 16, 96, 2, (1, 4)), (9, 13, 24, 144, 1, (1, 3)), (5, 5, 96, 576, 2, (1, 40)),
             (1, 1, 64, 72, 1, (1, 7)), (3, 3, 40, 40, 2, (2,)), (4, 254, 40, 16, 1, (1, 2)), (13, 61, 136, 200, 2, (1, 3)), (29, 31, 192, 24, 1, (1, 3)), (34, 34, 16, 96, 2, (2, 33))]


@pytest.mark.parametrize("geom", XDW_GEOMS)
def test_expand_and_depthwise_in_one_launch(geom):
    H, W, cin, hidden, stride, batches = geom
    bmax = batches[-1]
    rng = wl._rng(H + hidden, 927)
    layers = [wl._conv(rng, wl.OP_CONV, cin, hidden, 1, 1, 0, wl.ACT_RELU6, bf16=True), wl._conv(rng, wl.OP_DWCONV, hidden, hidden, 3, stride, 1, wl.ACT_RELU6, bf16=True)]
    layers[0].bias = layers[0].bias + 0.25          # outside the image the hidden map is zero, not act(bias)
    fw, fb = wl._head(rng, hidden, 5, 1.0, True)
    spec = wl.Model("xdw", "bf16", H, W, cin, [wl.Stage(layers, 5, fw, fb, 2.0, False)], bmax)
    run = util.GpuRunner(spec)
    m, out = run.m, run.bufs[0]
    x = wl.random_features((bmax, H, W, cin), seed=4, bf16=True, relu=False)
    xd = eb.to_device("bf16", x)
    first = None
    for B in batches:
        assert [pl["launches"] for pl in m.plan(0, B)] == [1, 0]
        m.stage_run(0, xd[:B], B, out, run.ws)
        torch.cuda.synchronize()
        m.check()
        got = out.features_out[:B].clone()
        if first is None:
            first = got
        assert torch.equal(got[: len(first)], first)     # alone or in a batch, other bands: the same bits
    hid = torch.empty((bmax, H, W, hidden), dtype=torch.bfloat16, device="cuda")
    apart = torch.empty_like(out.features_out[:bmax])
    m.layer_run(0, 0, xd, None, bmax, hid, run.ws)
    m.layer_run(0, 1, hid, None, bmax, apart, run.ws)
    torch.cuda.synchronize()
    if cin > 32:
        assert torch.equal(got, apart)
    o = eo.run_layers(spec, 0, x)
    # the bar of a chain of layers: a hidden value that rounds the other way moves by 2^-8 of itself, and the outputs that sum it with it,
    # so an element is off by a few 2^-8 of the largest, whatever its own size
    assert np.max(np.abs(got.float().cpu().numpy() - o)) <= 2.0 ** -6 * np.max(np.abs(o))
    m.set_layer_variant(0, 0, 1, 1, 4)      # a table entry: apart again, at every batch
    assert [pl["launches"] for pl in m.plan(0, batches[0])] == [1, 1]
    m.stage_run(0, xd, bmax, out, run.ws)
    torch.cuda.synchronize()
    assert torch.equal(out.features_out[:bmax], apart)
    run.check_guards()


# The expand + depthwise launch against the two layers run apart, narrow inputs, whose pixels are grouped apart (cin 8 to 32): channels that
# are whole K steps of 16 and such that are not, maps of an even and an odd number of pixels.  The depthwise layer hands its input on, so every
# hidden value shows; enough of them that K steps starting elsewhere would round some the other way.  H, W, cin, hidden, stride, batch
XDW_NARROW = [(28, 28, 8, 48, 1, 32), (16, 34, 16, 96, 2, 32), (34, 34, 24, 144, 1, 64), (28, 28, 24, 144, 1, 64), (33, 33, 24, 144, 2, 3), (28, 28, 32, 192, 1, 32), (28, 28, 24, 72, 1, 8),
              (12, 12, 24, 40, 1, 8)]


@pytest.mark.parametrize("geom", XDW_NARROW)
def test_expand_and_depthwise_of_narrow_layers_give_the_bits_of_the_layers_apart(geom):
    H, W, cin, hidden, stride, B = geom
    rng = wl._rng(W + hidden, 931)
    layers = [wl._conv(rng, wl.OP_CONV, cin, hidden, 1, 1, 0, wl.ACT_NONE, bf16=True), wl._conv(rng, wl.OP_DWCONV, hidden, hidden, 3, stride, 1, wl.ACT_NONE, bf16=True)]
    layers[1].weight = np.zeros_like(layers[1].weight)
    layers[1].weight[:, 1, 1, :] = 1.0
    layers[1].scale = layers[1].bias = None
    fw, fb = wl._head(rng, hidden, 5, 1.0, True)
    spec = wl.Model("xdw", "bf16", H, W, cin, [wl.Stage(layers, 5, fw, fb, 2.0, False)], B)
    run = util.GpuRunner(spec)
    m, out = run.m, run.bufs[0]
    assert [pl["launches"] for pl in m.plan(0, B)] == [1, 0]
    xd = eb.to_device("bf16", wl.random_features((B, H, W, cin), seed=6, bf16=True, relu=False))
    m.stage_run(0, xd, B, out, run.ws)
    torch.cuda.synchronize()
    m.check()
    fused = out.features_out[:B].clone()
    hid = torch.empty((B, H, W, hidden), dtype=torch.bfloat16, device="cuda")
    apart = torch.empty_like(fused)
    m.layer_run(0, 0, xd, None, B, hid, run.ws)
    m.layer_run(0, 1, hid, None, B, apart, run.ws)
    torch.cuda.synchronize()
    assert torch.equal(fused, apart)
    # entries for CTA pairs are taken as for grouped pixels, whatever the kernel behind them
    group = max(g for g in range(1, 64 // cin + 1) if H * W % g == 0)
    mask = (1 if group * hidden > 128 else 0) | (2 if group * hidden > 64 else 0)
    assert m.layer_config(0, 0, B)["tensor_core"] == mask
    for v in [v for v in (1, 2) if mask >> (v - 1) & 1] + [4]:
        m.set_layer_variant(0, 0, B, B, v)
        m.stage_run(0, xd, B, out, run.ws)
        torch.cuda.synchronize()
        m.check()
        assert torch.equal(out.features_out[:B], fused)
    m.set_layer_variant(0, 0, B, B, 0)
    assert [pl["launches"] for pl in m.plan(0, B)] == [1, 0]
    m.set_stage_kernel(True)         # multi-layer launches take single layers
    assert [pl["launches"] for pl in m.plan(0, B)] == [1, 1]
    m.stage_run(0, xd, B, out, run.ws)
    torch.cuda.synchronize()
    m.check()
    assert torch.equal(out.features_out[:B], fused)
    run.check_guards()


# Sums of negative zeros, sign and all: the ranges of a layer start from the same zero on every route (clusters of CTAs, one CTA per tile,
# the one-wave kernel, CTA pairs): H, W, cin, cout, ranges, batch
@pytest.mark.parametrize("geom", [(7, 7, 128, 128, 3, 4), (7, 7, 128, 256, 2, 40)])
def test_k_ranges_give_the_same_zero_on_every_route(geom):
    H, W, cin, cout, ranges, B = geom
    spec = util.single_layer_model("bf16", H, W, cin, cout, 3, 1, 1, wl.ACT_NONE, False, seed=3, max_batch=B)
    l = spec.stages[0].layers[0]
    l.weight, l.scale, l.bias = -np.abs(l.weight), None, np.full(cout, -0.0, dtype=np.float32)
    m = eb.EEModel(spec)
    m.set_layer_splits(0, 0, ranges)
    ws = m.workspace()
    x = wl.random_features((B, H, W, cin), seed=3, bf16=True)
    x[: (B + 1) // 2] = 0.0
    xd = eb.to_device("bf16", x)
    got = []
    for variant in (3, 4, 0, 1 if cout > 128 else 2):
        m.set_layer_variant(0, 0, 1, B, variant)
        out = torch.empty((B, H, W, cout), dtype=torch.bfloat16, device="cuda")
        m.layer_run(0, 0, xd, None, B, out, ws)
        torch.cuda.synchronize()
        m.check()
        got.append(out.view(torch.int16))
    assert all(torch.equal(g, got[0]) for g in got)


# What keeps the last layer from storing to features_out: its output is read inside the stage, or features_out lies in the stage's input or
# in the workspace, where the last layer still reads: a 3x3 layer over several waves of tiles, whose neighbours would be overwritten.  The
# survivors are the same rows as in a buffer of its own.
@pytest.mark.parametrize("dtype", ["bf16", "f32"])
@pytest.mark.parametrize("where", ["read inside", "residual inside", "input", "workspace"])
def test_survivors_are_gathered_where_features_out_cannot_take_the_output(dtype, where):
    inside = where in ("read inside", "residual inside")
    B, hw, c = 19, 6 if inside else 56, 64
    rng = wl._rng(c, 933)
    bf16 = dtype == "bf16"

    def layer(k, **kw):
        return wl._conv(rng, wl.OP_CONV, c, c, k, 1, k // 2, wl.ACT_RELU, bf16=bf16, **kw)

    from_input = dict(input_from=wl.FROM_STAGE_INPUT)
    layers = [layer(1), layer(3, **(from_input if where in ("input", "residual inside") else {}), **(dict(residual_from=0) if where == "residual inside" else {}))]
    fw, fb = wl._head(rng, c, 5, 1.0, bf16)
    spec = wl.Model("gathered", dtype, hw, hw, c, [wl.Stage(layers, 5, fw * 0.0, fb, 0.9, False, out_layer=0 if inside else 1)], B)
    run = util.GpuRunner(spec)
    m, out, ws = run.m, run.bufs[0], run.ws
    xd = eb.to_device(dtype, wl.random_features((B, hw, hw, c), seed=3, bf16=bf16))
    want, hid = torch.empty_like(out.features_out), torch.empty_like(out.features_out)
    m.layer_run(0, 0, xd, None, B, want if inside else hid, ws)
    if not inside:
        m.layer_run(0, 1, xd if where == "input" else hid, None, B, want, ws)
    xs = xd.clone()
    if where == "input":
        out.features_out = xs
    elif where == "workspace":       # its first slot, the hidden layer's
        out.features_out = ws[: want.numel() * want.element_size()].view(want.dtype).view(want.shape)
    out._struct = None
    for leave in (np.zeros(B, bool), np.arange(B) % 3 == 0, np.arange(B) > 4, np.ones(B, bool)):
        xs.copy_(xd)
        shift = torch.as_tensor(leave.astype(np.float32) * 30.0, device="cuda")
        m.stage_run(0, xs, B, out, ws, None, shift, torch.zeros(B, dtype=torch.int32, device="cuda"))
        torch.cuda.synchronize()
        stay = np.nonzero(~leave)[0]
        n = int(out.n_surv_dev[0])
        assert n == len(stay) and np.array_equal(out.survivor_idx[:n].cpu().numpy(), stay)
        assert torch.equal(out.features_out[:n], want[torch.as_tensor(stay, device="cuda")])
    m.check()
    run.check_guards()
