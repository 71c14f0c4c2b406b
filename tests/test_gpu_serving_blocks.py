"""The building blocks of FluidServer called one by one, with the server's own buffers and with a caller's."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_2209_13443_b200 import binding as eb
from paper_2209_13443_b200 import workloads as wl
from paper_2209_13443_b200.serving import FluidServer, _Clock

pytestmark = pytest.mark.gpu


def _run(server, pool, rows, members, feat, ids, bufs):
    out = server._result(128)
    server.form_batch(pool, rows, members, feat, ids)
    stay = server.run_stage(0, feat, ids, members, bufs, _Clock(lambda s, n: 1e-3), out)
    torch.cuda.synchronize()
    n = len(members)
    return (stay, feat[:n].clone(), ids[:n].clone(), bufs[0].features_out[: len(stay)].clone(), bufs[0].ids_out[: len(stay)].clone(),
            [out[k].tolist() for k in ("finish", "exit_stage", "pred")])


def _same(a, b):
    return all(torch.equal(x, y) if isinstance(x, torch.Tensor) else x == y for x, y in zip(a, b))


def test_blocks_take_the_callers_ids_and_stage_buffers():
    spec = wl.tiny_ee_cnn(seed=0)
    server = FluidServer(spec)
    pool = eb.to_device("f32", wl.make_input(spec, 16, seed=2))
    rows, members = [5, 1, 3, 15, 0, 2, 9], [100, 7, 42, 3, 127, 0, 64]
    own = _run(server, pool, rows, members, server.in_act, server.ids_act, server.act)
    assert own[2].tolist() == members and 0 < len(own[0]) < len(members)      # some leave, some stay
    ids = torch.full((spec.max_batch,), -1, dtype=torch.int32, device="cuda")
    feat = torch.empty_like(server.in_act)
    pinned = [eb.StageBuffers(server.m, s, pinned_decisions=True) for s in range(server.n_stages)]
    device = [eb.StageBuffers(server.m, s) for s in range(server.n_stages)]
    for bufs in (server.act, pinned, device):
        assert _same(_run(server, pool, rows, members, feat, ids, bufs), own)
    assert ids[len(members):].tolist() == [-1] * (spec.max_batch - len(members))
    wide = torch.empty(spec.max_batch, dtype=torch.int64, device="cuda")       # ids as the caller holds them
    server.form_batch(pool, rows, members, feat, wide)
    assert wide[: len(members)].tolist() == members


def test_batches_formed_one_behind_the_other_in_the_callers_buffers():
    spec = wl.tiny_ee_cnn(seed=0)
    server = FluidServer(spec)
    pool = eb.to_device("f32", wl.make_input(spec, 16, seed=2))
    batches = [([(7 * k + j) % 16 for j in range(1 + k % 8)], [10 * k + j for j in range(1 + k % 8)]) for k in range(12)]
    bufs = [(torch.empty_like(server.in_act), torch.empty(spec.max_batch, dtype=torch.int32, device="cuda")) for _ in batches]
    torch.cuda.synchronize()
    for (rows, members), (feat, ids) in zip(batches, bufs):       # no stage in between: nothing waits for an upload but form_batch
        server.form_batch(pool, rows, members, feat, ids)
    torch.cuda.synchronize()
    for (rows, members), (feat, ids) in zip(batches, bufs):
        assert ids[: len(members)].tolist() == members and torch.equal(feat[: len(rows)], pool[rows])
    assert np.isfinite(feat[: len(rows)].cpu().numpy()).all()


def test_a_count_that_disagrees_with_the_decisions_is_an_error():
    spec = wl.tiny_ee_cnn(seed=0)
    server = FluidServer(spec)
    pool = eb.to_device("f32", wl.make_input(spec, 16, seed=2))
    server.thr[0] = (np.float32(2.0), False)                      # the host's copy of the threshold alone: nobody would leave
    with pytest.raises(RuntimeError, match="stay by the device's count"):
        _run(server, pool, [5, 1, 3, 15, 0, 2, 9], [0, 1, 2, 3, 4, 5, 6], server.in_act, server.ids_act, server.act)


def test_a_trace_runs_on_the_current_stream_and_blocks_on_theirs():
    spec = wl.tiny_ee_cnn(seed=0)
    server = FluidServer(spec)
    pool = eb.to_device("f32", wl.make_input(spec, 16, seed=2))
    arrivals, image_of = wl.poisson_arrivals(1, 20, 2000.0), [3 * i % 16 for i in range(20)]
    torch.cuda.synchronize()
    side, got = torch.cuda.Stream(), []
    for ctx in (torch.cuda.default_stream(), side):
        with torch.cuda.stream(ctx):
            r = server.serve(arrivals, image_of, pool, lambda s, n: 1e-3)
            got.append([r[k].tolist() for k in ("finish", "exit_stage", "pred")])
            assert server.stream is None
    assert got[0] == got[1]
    with pytest.raises(ValueError):
        server.serve(arrivals, image_of, pool, slo=1.0)
    assert server.stream is None
    own = _run(server, pool, [5, 1, 3], [0, 1, 2], server.in_act, server.ids_act, server.act)
    with torch.cuda.stream(side):
        assert _same(_run(server, pool, [5, 1, 3], [0, 1, 2], server.in_act, server.ids_act, server.act), own)
