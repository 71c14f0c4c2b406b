"""Timed cases of the early-exit stage executor: what programs on top of it call, over the sizes they call it with.

A case is one call sequence through the public entry points (``EEModel``, ``StageBuffers``, ``gather_survivors``,
``FluidServer``), described by a dict of plain values:

  kind "pass"   a batch of requests through every exit: ``batch_refill`` puts the arrivals into the batch buffer, then
                either the library drives the stages (``run_until_exit``) or the caller does, stage by stage
                (``stage_run`` and ``wait_count``), as a scheduler with its own policy would.
  kind "head"   ``exit_head`` alone, for a caller with a backbone of its own.
  kind "merge"  a preemption point: the survivors parked at a stage boundary are compacted (``gather_survivors``) and
                the samples that caught up are appended behind them (``batch_refill``).
  kind "serve"  ``FluidServer.serve``: a request trace on a virtual clock, with preemption and merging.

Networks, image sizes and batch limits are those of ``workloads.py`` and the benchmark.  Who leaves at which exit is
forced by logit shifts on flat heads (the benchmark's exit-rate mode), so the batch sizes of a pass are a property of
the case and no sample sits at its threshold.  The model and the buffers of a pass (batch, workspace, stage outputs) are
kept from call to call, as a server keeps them, and shared by the states of a case; a state has its own inputs, and for
"head" and "merge" its own outputs.
"""
import dataclasses

import numpy as np
import torch

from paper_2209_13443_b200 import binding as eb
from paper_2209_13443_b200 import workloads as wl
from paper_2209_13443_b200.serving import FluidServer

_FLAT = 0.01      # head scale at which only forced shifts decide an exit
_SHIFT = 16.0     # what a forced sample gets on one logit


def _pass(name, net, batch, p=0.0, hw=224, bmax=64, driver="library", stream="own", dtype="bf16", classes=1000):
    return {"name": name, "kind": "pass", "net": net, "dtype": dtype, "hw": hw, "classes": classes, "bmax": bmax, "batch": batch,
            "p": p, "driver": driver, "stream": stream}


def listed():
    return [
        # the smallest model (fp32) at a full batch, by a program that never chose a stream: launch latency and host path
        _pass("tiny f32 b8", "tiny", 8, 0.25, hw=32, bmax=8, stream="default", dtype="f32", classes=10),
        # one request alone in a server built for 64, never leaving early: the latency a lone user sees
        _pass("resnet50 b1", "resnet50", 1),
        # a handful of requests under a scheduler that drives the stages itself
        _pass("resnet50 b7 caller", "resnet50", 7, 0.3, driver="caller"),
        # the benchmark: a full batch that shrinks by about a third at every exit
        _pass("resnet50 b64 caller", "resnet50", 64, 0.3, driver="caller"),
        # a full batch in which nobody leaves: the largest amount of work a pass can be
        _pass("resnet50 b64 nobody leaves", "resnet50", 64),
        # images that are not the benchmark's size, a ragged batch, the default stream
        _pass("resnet50 b21 161px", "resnet50", 21, 0.2, hw=161, stream="default"),
        # the second benchmark network at its batch limit
        _pass("mobilenetv2 b32 caller", "mobilenetv2", 32, 0.25, bmax=32, driver="caller"),
        # factorised 1x7 / 7x1 filters
        _pass("tower b13", "tower", 13, 0.25, hw=68, bmax=32),
        # the fp32 model on small images: the path for callers who ask for 1e-5
        _pass("resnet50 f32 b6 64px", "resnet50", 6, 0.3, hw=64, bmax=6, dtype="f32", classes=100),
        # an exit decision on the caller's own feature map
        {"name": "head b37 28x28x512", "kind": "head", "stage": 1, "batch": 37, "rows": 784, "stream": "own"},
        # a trace of requests through the scheduler of the paper (fp32 model, exits by confidence): its host loop and the small calls
        {"name": "serve 48 requests", "kind": "serve", "requests": 48, "rate": 2000.0, "stream": "own"},
        # a preemption point at the first exit: 41 of 64 stay, 23 caught up
        {"name": "merge 41+23 56x56x256", "kind": "merge", "net": "resnet50", "boundary": 1, "bmax": 64, "stay": 41, "join": 23, "stream": "own"},
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(lo * (hi / lo) ** rng.random()))))


def draw(rng):
    r = rng.random()
    p, driver, stream = rng.choice([0.0, 0.1, 0.25, 0.4]), rng.choice(["library", "caller"]), rng.choice(["own", "own", "default"])
    kw = dict(driver=driver, stream=stream)
    if r < 0.38:
        c = _pass("", "resnet50", _log_int(rng, 1, 64), p, hw=rng.choice([224, _log_int(rng, 96, 224)]), **kw)
    elif r < 0.58:
        c = _pass("", "mobilenetv2", _log_int(rng, 1, 32), p, hw=rng.choice([224, _log_int(rng, 96, 224)]), bmax=32, **kw)
    elif r < 0.68:
        c = _pass("", "tower", _log_int(rng, 1, 32), p, hw=_log_int(rng, 44, 100), bmax=32, **kw)
    elif r < 0.74:
        c = _pass("", "tiny", rng.randint(1, 8), p, hw=rng.randint(24, 40), bmax=8, dtype="f32", classes=10, **kw)
    elif r < 0.80:
        c = _pass("", "resnet50", rng.randint(1, 6), p, hw=rng.randint(33, 64), bmax=6, dtype="f32", classes=100, **kw)
    elif r < 0.89:
        stage = rng.randint(0, 3)
        c = {"kind": "head", "stage": stage, "batch": _log_int(rng, 1, 64), "rows": rng.randint(*[(600, 3136), (160, 784), (40, 196), (9, 49)][stage]),
             "stream": stream}
    elif r < 0.96:
        net = rng.choice(["resnet50", "mobilenetv2"])
        stay = rng.randint(1, 31)
        c = {"kind": "merge", "net": net, "boundary": rng.randint(1, 3), "bmax": 64 if net == "resnet50" else 32, "stay": stay,
             "join": rng.randint(1, 32 - stay), "stream": stream}
    else:
        c = {"kind": "serve", "requests": rng.randint(24, 64), "rate": float(rng.randint(1000, 4000)), "stream": stream}
    c.pop("name", None)
    return c


# ----------------------------------------------------------------------------- what a program keeps

_specs = {}   # network description by (net, dtype, classes): weights do not depend on the image size or the batch limit
_kept = {}    # what the program of the case at hand keeps


def _spec(net, dtype, classes, hw, bmax):
    key = (net, dtype, classes)
    if key not in _specs:
        while len(_specs) >= 3:
            _specs.pop(next(iter(_specs)))
        if net == "resnet50":
            _specs[key] = wl.resnet50_ee(alphas=[_FLAT] * 4, n_classes=classes, dtype=dtype)
        elif net == "mobilenetv2":
            _specs[key] = wl.mobilenetv2_ee(alphas=[_FLAT] * 4, n_classes=classes, dtype=dtype)
        elif net == "tower":
            _specs[key] = wl.factorised_tower_ee(alphas=[_FLAT] * 2, n_classes=classes)
        elif net == "tiny":
            _specs[key] = wl.tiny_ee_cnn(alphas=(_FLAT,) * 3)
        else:
            _specs[key] = wl.tiny_ee_cnn()     # "tiny natural": exits by confidence
    return dataclasses.replace(_specs[key], in_h=hw, in_w=hw, max_batch=bmax)


def _case_spec(case):
    if case["kind"] == "pass":
        return _spec(case["net"], case["dtype"], case["classes"], case["hw"], case["bmax"])
    if case["kind"] == "head":
        return _spec("resnet50", "bf16", 1000, 224, 64)
    if case["kind"] == "merge":
        return _spec(case["net"], "bf16", 1000, 224, case["bmax"])
    return _spec("tiny natural", "f32", 10, 32, 8)


class _Kept:
    """Model, stream and buffers of a server: built at the first call for this kind of work, kept for the following ones."""

    def __init__(self, case, spec):
        self.stream = torch.cuda.Stream() if case["stream"] == "own" else torch.cuda.default_stream()
        self.model = m = eb.EEModel(spec)
        if case["kind"] == "pass":
            self.bufs = [eb.StageBuffers(m, s) for s in range(m.n_stages)]
            self.ws = m.workspace()
            self.batch = torch.empty((m.max_batch, spec.in_h, spec.in_w, spec.in_c), dtype=eb.torch_dtype(m.dtype), device="cuda")
            self.ids = torch.empty(m.max_batch, dtype=torch.int32, device="cuda")
        elif case["kind"] == "serve":
            self.server = FluidServer(spec, m)


def _keep(case):
    spec = _case_spec(case)
    key = (case["kind"], spec.name, spec.dtype, spec.in_h, spec.max_batch, case["stream"])
    if key not in _kept:
        _kept.clear()
        _kept[key] = _Kept(case, spec)
    return _kept[key]


def _sizes(case, n_stages):
    """Batch of every stage of a pass: a share p of the samples leaves at each early exit (driver "library": at the first)."""
    sizes = [case["batch"]]
    for s in range(n_stages - 1):
        p = case["p"] if case["driver"] == "caller" or s == 0 else 0.0
        sizes.append(max(1, sizes[-1] - int(round(p * sizes[-1]))))
    return sizes


def _images(n, hw, gen, dtype):
    """Images as workloads.make_input describes them (white noise plus a coarse 4x4 field), drawn on the device."""
    white = torch.randn((n, hw, hw, 3), generator=gen, device="cuda")
    at = torch.arange(hw, device="cuda") // -(-hw // 4)
    coarse = torch.randn((n, 4, 4, 3), generator=gen, device="cuda")[:, at][:, :, at]
    return ((white + coarse) * 0.5 ** 0.5).to(dtype)


# ----------------------------------------------------------------------------- states

def prepare(case, seed):
    kept = _keep(case)
    model, stream = kept.model, kept.stream
    gen = torch.Generator(device="cuda").manual_seed(seed)
    rng = np.random.default_rng(seed)
    td = eb.torch_dtype(model.dtype)
    st = {"kind": case["kind"], "model": model, "stream": stream}
    if case["kind"] == "pass":
        n_st, b = model.n_stages, case["batch"]
        sizes = _sizes(case, n_st)
        st.update(driver=case["driver"], n=b, x=_images(b, case["hw"], gen, td), x_ids=torch.randperm(1 << 16, generator=gen, device="cuda")[:b].int(),
                  ws=kept.ws, bufs=kept.bufs, batch=kept.batch, ids=kept.ids)
        # forced exits: at exit s a random sizes[s] - sizes[s + 1] of the sizes[s] samples leave
        st["forced"] = []
        for s in range(n_st):
            shift = np.zeros(sizes[s], dtype=np.float32)
            if s + 1 < n_st:
                shift[rng.permutation(sizes[s])[:sizes[s] - sizes[s + 1]]] = _SHIFT
            cls = rng.integers(0, case["classes"], sizes[s]).astype(np.int32)
            st["forced"].append((torch.from_numpy(shift).cuda(), torch.from_numpy(cls).cuda()))
        # pred is the argmax of logits and left out: the top of 1000 flat logits is often a near-tie
        st["out"] = {}
        for s, n in enumerate(sizes):
            o = st["bufs"][s]
            st["out"].update({f"conf{s}": o.conf[:n], f"logits{s}": o.logits[:n], f"mask{s}": o.exit_mask[:n], f"left{s}": o.n_surv_dev})
            if s + 1 < n_st:
                m = sizes[s + 1]
                st["out"].update({f"features{s}": o.features_out[:m], f"survivors{s}": o.survivor_idx[:m], f"ids{s}": o.ids_out[:m]})
    elif case["kind"] == "head":
        s, b, rows = case["stage"], case["batch"], case["rows"]
        c = model.query(s)["out_c"]
        o = eb.StageBuffers(model, s)
        left = torch.zeros(b, dtype=torch.bool, device="cuda")
        left[torch.randperm(b, generator=gen, device="cuda")[:int(0.3 * b)]] = True    # forced to leave
        st.update(stage=s, n=b, rows=rows, x=torch.randn((b, rows, c), generator=gen, device="cuda").abs_().to(td), buf=o,
                  scratch=torch.empty(model.exit_head_scratch_bytes(s) + 256, dtype=torch.uint8, device="cuda"),
                  shift=left.float() * _SHIFT, cls=torch.randint(0, 1000, (b,), generator=gen, device="cuda").int())
        m = b - int(0.3 * b) if s + 1 < model.n_stages else 0
        st["out"] = {"conf": o.conf[:b], "logits": o.logits[:b], "mask": o.exit_mask[:b], "left": o.n_surv_dev, "survivors": o.survivor_idx[:m]}
    elif case["kind"] == "merge":
        q = model.query(case["boundary"])
        shape, k, j, b = (q["in_h"], q["in_w"], q["in_c"]), case["stay"], case["join"], case["bmax"]
        st.update(boundary=case["boundary"], stay=k, join=j, row_bytes=q["in_bytes_per_sample"],
                  parked=torch.randn((b,) + shape, generator=gen, device="cuda").to(td), fresh=torch.randn((j,) + shape, generator=gen, device="cuda").to(td),
                  idx=torch.from_numpy(np.sort(rng.permutation(b)[:k]).astype(np.int32)).cuda(), cnt=torch.tensor([k], dtype=torch.int32, device="cuda"),
                  merged=torch.empty((b,) + shape, dtype=td, device="cuda"), ids=torch.arange(b, dtype=torch.int32, device="cuda"),
                  fresh_ids=torch.randperm(1 << 16, generator=gen, device="cuda")[:j].int())
        st["out"] = {"merged": st["merged"][:k + j], "ids": st["ids"][:k + j]}
    else:
        n = case["requests"]
        st.update(server=kept.server, arrivals=wl.poisson_arrivals(seed, n, case["rate"]), image_of=rng.integers(0, 32, n).tolist(),
                  pool=_images(32, 32, gen, td))
    stream.wait_stream(torch.cuda.current_stream())
    return st


def _stage_time(stage, batch):   # the virtual clock of a trace: seconds a stage takes at a batch size
    return 2e-4 * (stage + 1) + 3e-5 * batch


def run(st):
    m, stream = st["model"], st["stream"]
    if st["kind"] == "pass":
        bufs, ws, feat, ids = st["bufs"], st["ws"], st["batch"], st["ids"]
        _, n = m.batch_refill(0, feat, ids, 0, st["x"], st["x_ids"], st["n"], stream=stream)
        if st["driver"] == "library":
            shift, cls = st["forced"][0]
            m.run_until_exit(0, feat, n, bufs, ws, ids, shift, cls, stream=stream)
            return st["out"]
        last = m.n_stages - 1
        for s in range(m.n_stages):
            o, (shift, cls) = bufs[s], st["forced"][s]
            o.arm_count()
            m.stage_run(s, feat, n, o, ws, ids, shift, cls, stream=stream)
            if s == last:
                break
            n = o.wait_count()
            if n == 0:
                break
            feat, ids = o.features_out, o.ids_out
        return st["out"]
    if st["kind"] == "head":
        m.exit_head(st["stage"], st["x"], st["n"], st["rows"], st["buf"], st["scratch"], st["shift"], st["cls"], stream=stream)
        return st["out"]
    if st["kind"] == "merge":
        eb.gather_survivors(st["parked"], st["row_bytes"], st["idx"], st["cnt"], st["stay"], st["merged"], stream=stream)
        m.batch_refill(st["boundary"], st["merged"], st["ids"], st["stay"], st["fresh"], st["fresh_ids"], st["join"], stream=stream)
        return st["out"]
    with torch.cuda.stream(stream):
        r = st["server"].serve(st["arrivals"], st["image_of"], st["pool"], _stage_time)
    return {"finish": r["finish"], "exit": r["exit_stage"], "pred": r["pred"], "preemptions": r["preemptions"], "stage launches": len(r["launches"])}


# ----------------------------------------------------------------------------- what a pass cannot do without

def work(case):
    """Inputs read once (images, weights of the stages reached), outputs written once; multiply-adds of the samples at every stage."""
    spec = _case_spec(case)
    shapes = wl.stage_shapes(spec)
    es = 2 if spec.dtype == "bf16" else 4

    def elems(shape):
        return int(np.prod(shape))

    def stage(s):   # (weight elements, flops per sample) of a stage and its head
        w = f = 0
        for l, o in zip(spec.stages[s].layers, shapes[s]["layers"]):
            if l.op != wl.OP_MAXPOOL:
                k = l.kh * l.kw * (l.cin // l.groups)
                w, f = w + l.cout * k, f + 2.0 * elems(o) * k
        fc = spec.stages[s].n_classes * shapes[s]["out"][2]
        return w + fc, f + 2.0 * fc

    if case["kind"] == "pass":
        sizes = _sizes(case, len(spec.stages))
        byt, flops = 2 * case["batch"] * elems(shapes[0]["in"]) * es, 0.0     # arrivals read, batch buffer written
        for s, n in enumerate(sizes):
            w, f = stage(s)
            byt, flops = byt + w * es + 4 * n * spec.stages[s].n_classes, flops + n * f
            if s + 1 < len(sizes):
                byt += sizes[s + 1] * elems(shapes[s]["out"]) * es
        return {"bytes": byt, "flops": flops}
    if case["kind"] == "head":
        c, k = shapes[case["stage"]]["out"][2], 1000
        return {"bytes": case["batch"] * (case["rows"] * c * es + 4 * k) + k * c * es, "flops": case["batch"] * c * (case["rows"] + 2.0 * k)}
    if case["kind"] == "merge":
        return {"bytes": 2 * (case["stay"] + case["join"]) * elems(shapes[case["boundary"]]["in"]) * es, "flops": 0.0}
    w, f = stage(0)    # every request runs at least the first stage
    return {"bytes": case["requests"] * elems(shapes[0]["in"]) * es + w * es, "flops": case["requests"] * f}


def tolerance(case):
    if case["kind"] == "merge":
        return "exact"
    if case["kind"] == "serve":
        return {"rel": 1e-9, "max": 1e-6, "differ": 0.0}     # times of a virtual clock; exits, classes and batches are whole numbers
    if case["kind"] == "head" or case["dtype"] == "f32":
        return {"rel": 1e-5, "max": 1e-3}
    return {"rel": 1e-2, "max": 0.2}                           # up to 52 layers, each rounded to bf16
