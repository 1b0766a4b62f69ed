"""Performance cases of the library: what a user's program has it do, through
the public entry points of ``paper_2009_04509_gb300.emtk``.

A case is a dict of plain values:

  op         "infer"    one emtk_infer per plane
             "batch"    emtk_infer_batch over all planes
             "host"     emtk_infer_batch_host over all planes (pinned host buffers)
             "patches"  emtk_infer_patches on pre-cut patches
             "cut"      emtk_extract_patches, one call per plane
             "find"     emtk_find_hits over all planes
  precision  of the context: "fp32", "tf32", "bf16", "fp16" or "fp8"
  logits     contexts created with debug_logits: 8 columns (4 scores, 4 logits)
  planes     number of planes; plane i has entry i % len(wires) of wires, a list as text
  wires, nticks, pad      plane shapes; rows are nticks rounded up to 4, plus 4 * pad
  hits       per plane, as wires
  tracks, showers, michel, shower_share, michel_share   what a plane holds
  fmt        of the patches ("cut")
  threshold  ("find")
  patches    ("patches")

Inputs follow the recipe of ``synth`` (the repository's stand-in for the
detector data), drawn on the GPU: Gaussian noise of sigma 3 plus pulses of
sigma 3 ticks and amplitude U(20, 200) along straight tracks, in cone-shaped
showers and along short Michel-like segments; pre-cut patches are 70 % zeros,
else lognormal(2, 1).  The weights are the He-normal ones of seed 0.
"""
from __future__ import annotations

import functools
import math
import weakref

import torch

from paper_2009_04509_gb300 import emtk, synth

DEV = "cuda"
NET_FLOPS = 28_444_416       # conv, dense-1, dense-2 and heads of one hit
W1_VALUES = 92_928 * 128     # dense-1 weights, read once by every pass of the network
W1_BYTES = {"fp32": 4, "tf32": 4, "bf16": 2, "fp16": 2, "fp8": 1}
WINDOW_BYTES = 48 * 48 * 6 * 4
FIND_ROOM = 64               # rows per wire of a hit-finding output (about 11 are used on the full event)


def _planes(op, precision, **kw):
    case = dict(op=op, precision=precision, logits=False, planes=1, wires="480", nticks=6000, pad=0, hits="256",
                tracks=5, showers=0, michel=0, shower_share=0.0, michel_share=0.0)
    case.update(kw)
    return case


# The workloads of the repository's benchmark and tests.
_APA = dict(planes=3, wires="800 800 480", hits="7692 7692 4616", tracks=30, showers=5, shower_share=0.3)
_EVENT = dict(planes=18, wires="800 800 960", hits="3125 3125 3750", tracks=30, showers=5, michel=10,
              shower_share=0.3, michel_share=0.1)


def listed():
    return [
        # one collection plane of a small request: latency of a single call
        dict(_planes("infer", "bf16"), name="plane_256_bf16"),
        # the same at the paper's own precision
        dict(_planes("infer", "fp32"), name="plane_256_fp32"),
        # an inference-server batch of pre-cut patches (the paper's larger mean batch, an odd size)
        dict(op="patches", precision="bf16", logits=True, patches=1693, name="patches_1693_bf16"),
        # the same batch at the paper's own precision
        dict(op="patches", precision="fp32", logits=False, patches=1693, name="patches_1693_fp32"),
        # one detector module (APA), a call per plane as its planes come in
        dict(_planes("infer", "bf16", logits=True, **_APA), name="apa_bf16"),
        # the same module in one batched call, at fp32 accuracy on the tensor cores
        dict(_planes("batch", "tf32", **_APA), name="apa_tf32"),
        # ... and in fp32
        dict(_planes("batch", "fp32", **_APA), name="apa_fp32"),
        # a full event of 18 planes in one batched call: the benchmark's workload
        dict(_planes("batch", "bf16", logits=True, **_EVENT), name="event_bf16"),
        # the same with the 8-bit dense layer
        dict(_planes("batch", "fp8", logits=True, **_EVENT), name="event_fp8"),
        # an event that arrives in host memory, copies included
        dict(_planes("host", "bf16", logits=True, **_EVENT), name="event_host_bf16"),
        # the patches of one plane for another network or for training
        dict(_planes("cut", "fp32", fmt="f32", wires="800", hits="7692", tracks=30, showers=5, shower_share=0.3),
             name="cut_plane_f32"),
        # hit finding on a full event, at five sigma of the noise
        dict(_planes("find", "bf16", threshold=15.0, **_EVENT), name="find_event"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _text(numbers):
    return " ".join(str(n) for n in numbers)


def draw(rng):
    """Any entry point and precision; 1 to 18 planes of 24 to 960 wires and 300
    to 6000 ticks; 1 to 60,000 hits or patches (20,000 at the fp32 accuracies,
    whose hits cost more)."""
    op = rng.choice(["infer", "batch", "batch", "host", "patches", "patches", "cut", "find"])
    precision = rng.choice(["bf16", "bf16", "fp16", "fp8", "tf32", "fp32"])
    logits = precision not in ("fp32", "tf32")
    most = 20_000 if precision in ("fp32", "tf32") else 60_000
    if op == "patches":
        return dict(op=op, precision=precision, logits=logits, patches=_log(rng, 1, most))
    planes = _log(rng, 1, 4 if op in ("infer", "cut") else 18)
    wires = [_log(rng, 24, 960) for _ in range(min(planes, 3))]
    nticks = _log(rng, 300, 6000)
    hits = [max(1, _log(rng, 1, 20_000 if op == "cut" else most) // planes) for _ in wires]
    case = _planes(op, precision, logits=logits, planes=planes, wires=_text(wires), nticks=nticks,
                   pad=rng.choice([0, 0, 1, 5]), hits=_text(hits), tracks=rng.randint(2, 30),
                   showers=rng.randint(1, 5), michel=rng.randint(1, 10),
                   shower_share=rng.choice([0.0, 0.3]), michel_share=rng.choice([0.0, 0.1]))
    if op == "cut":
        case["precision"], case["logits"] = "bf16", False  # the format is the call's, not the context's
        case["fmt"] = rng.choice(["f32", "bf16", "fp16"])
    if op == "find":
        case["precision"], case["logits"] = "bf16", False
        case["threshold"] = round(rng.uniform(10.0, 30.0), 2)
    return case


# ------------------------------------------------------------------ inputs
def _uniform(g, n, lo, hi):
    return torch.rand(n, generator=g, device=DEV, dtype=torch.float64) * (hi - lo) + lo


def _segments(w0, t0, w1, t1, nwires, nticks):
    """Wires crossed by segments (w0, t0)-(w1, t1) and the tick on each."""
    ws = torch.arange(nwires, device=DEV, dtype=torch.float64)[None, :]
    on = (ws >= torch.minimum(w0, w1)[:, None]) & (ws <= torch.maximum(w0, w1)[:, None])
    t = t0[:, None] + (ws - w0[:, None]) * ((t1 - t0) / (w1 - w0))[:, None]
    on &= (t >= 0) & (t <= nticks - 1)
    return ws.expand_as(t)[on].long(), t[on]


def _plane(g, nwires, nticks, ld, nhits, case):
    adc = torch.zeros(nwires, ld, device=DEV)
    adc[:, :nticks] = 3.0 * torch.randn(nwires, nticks, generator=g, device=DEV)
    n = case["tracks"]
    lines = [_segments(_uniform(g, n, 0, nwires), _uniform(g, n, 0, nticks), _uniform(g, n, 0, nwires),
                       _uniform(g, n, 0, nticks), nwires, nticks)]
    if case["michel"]:
        n = case["michel"]
        w, t = _uniform(g, n, 0, nwires), _uniform(g, n, 0, nticks)
        angle, length = _uniform(g, n, 0, 2 * math.pi), _uniform(g, n, 5, 20)
        lines.append(_segments(w, t, w + length * torch.cos(angle), t + 6 * length * torch.sin(angle), nwires, nticks))
    pw, pt = torch.cat([w for w, _ in lines]), torch.cat([t for _, t in lines])
    shower = int(round(nhits * case["shower_share"])) if case["showers"] else 0
    michel = int(round(nhits * case["michel_share"])) if case["michel"] else 0
    hw, ht = [], []
    for (w, t), k in zip(lines, (nhits - shower - michel, michel)):
        if k and w.numel() == 0:  # no line crosses a wire: hits anywhere
            w = torch.randint(0, nwires, (k,), generator=g, device=DEV)
            t = _uniform(g, k, 0, nticks - 1)
        if k:
            at = torch.randint(0, w.numel(), (k,), generator=g, device=DEV)
            hw.append(w[at])
            ht.append(t[at])
    if shower:
        k = case["showers"]
        which = torch.randint(0, k, (shower,), generator=g, device=DEV)
        wa, ta = _uniform(g, k, 0, nwires)[which], _uniform(g, k, 0, nticks)[which]
        angle, depth = _uniform(g, k, 0, 2 * math.pi)[which], _uniform(g, k, 50, 200)[which] * _uniform(g, shower, 0, 1)
        side = torch.randn(shower, generator=g, device=DEV, dtype=torch.float64) * depth * math.tan(0.2)
        w = (wa + depth * torch.cos(angle) - side * torch.sin(angle)).round().long().clamp(0, nwires - 1)
        t = (ta + 6 * (depth * torch.sin(angle) + side * torch.cos(angle))).clamp(0, nticks - 1)
        pw, pt = torch.cat([pw, w]), torch.cat([pt, t])
        hw.append(w)
        ht.append(t)
    # pulses, cut at 4 sigma; multiples of 2^-8, so that their sum does not depend on its order
    amp = _uniform(g, pw.numel(), 20, 200)
    t = pt.floor().long()[:, None] + torch.arange(-12, 14, device=DEV)[None, :]
    off = t - pt[:, None]
    val = (amp[:, None] * torch.exp(-0.5 * (off / 3.0) ** 2) * 256).round() / 256
    keep = (off.abs() <= 12) & (t >= 0) & (t < nticks)
    pulses = torch.zeros(nwires * ld, device=DEV)
    pulses.index_add_(0, (pw[:, None] * ld + t)[keep], val[keep].float())
    adc += pulses.view(nwires, ld)
    hits = torch.stack([torch.cat(hw), torch.cat(ht).round().long()], 1).int()
    order = torch.randperm(nhits, generator=g, device=DEV)
    return adc, hits[order].contiguous()


def _shapes(case):
    """(nwires, ld, nhits) of every plane."""
    ld = (case["nticks"] + 3) // 4 * 4 + 4 * case["pad"]
    wires, hits = ([int(n) for n in case[k].split()] for k in ("wires", "hits"))
    return [(wires[i % len(wires)], ld, hits[i % len(hits)]) for i in range(case["planes"])]


def _inputs(case, seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    if case["op"] == "patches":
        shape = (case["patches"], 48, 48)
        on = torch.rand(shape, generator=g, device=DEV) < 0.3
        val = torch.exp(2.0 + torch.randn(shape, generator=g, device=DEV))
        return torch.where(on, val, torch.zeros_like(val))
    return [_plane(g, nw, case["nticks"], ld, nh, case) for nw, ld, nh in _shapes(case)]


@functools.lru_cache(maxsize=1)
def _weights():
    return synth.he_normal_weights(0)


class _Context:
    """A context that lives as long as the state that holds it."""

    def __init__(self, precision, logits):
        self.handle = emtk.emtk_create(_weights(), precision=precision, debug_logits=logits)
        self._end = weakref.finalize(self, emtk.emtk_destroy, self.handle)


def prepare(case, seed):
    ctx = _Context(case["precision"], case["logits"])
    op, cols = case["op"], 8 if case["logits"] else 4
    state = {"case": case, "ctx": ctx}
    data = _inputs(case, seed)
    if op == "patches":
        state["patches"] = data
        state["out"] = torch.zeros(case["patches"], cols, device=DEV)
    elif op == "cut":
        dtype = {"f32": torch.float32, "bf16": torch.bfloat16, "fp16": torch.float16}[case["fmt"]]
        state["items"] = [(adc, hits, torch.zeros(hits.shape[0], 48, 48, device=DEV, dtype=dtype)) for adc, hits in data]
    elif op == "find":
        room = [adc.shape[0] * FIND_ROOM for adc, _ in data]
        hits = torch.zeros(sum(room), 2, device=DEV, dtype=torch.int32)
        info = torch.zeros(sum(room), 4, device=DEV, dtype=torch.int32)
        state["items"] = [(adc, case["nticks"], case["threshold"], h, i)
                          for (adc, _), h, i in zip(data, hits.split(room), info.split(room))]
        state["out"] = [hits, info[:, :2], info[:, 2:].view(torch.float32)]
    elif op == "host":
        # an event as it is read from one file: the planes back to back in one pinned buffer
        buf = torch.empty(sum(adc.numel() for adc, _ in data), pin_memory=True)
        state["items"], at = [], 0
        for adc, hits in data:
            plane = buf[at:at + adc.numel()].view_as(adc)
            plane.copy_(adc)
            at += adc.numel()
            state["items"].append((plane, case["nticks"], hits.cpu(),
                                   torch.zeros(hits.shape[0], cols, pin_memory=True)))
    else:
        state["items"] = [(adc, case["nticks"], hits, torch.zeros(hits.shape[0], cols, device=DEV))
                          for adc, hits in data]
    torch.cuda.synchronize()
    return state


def run(state):
    case, ctx = state["case"], state["ctx"].handle
    op = case["op"]
    if op == "patches":
        emtk.emtk_infer_patches(ctx, state["patches"], state["out"])
        return state["out"]
    items = state["items"]
    if op == "cut":
        for adc, hits, patches in items:
            emtk.emtk_extract_patches(ctx, adc, case["nticks"], hits, patches, fmt=case["fmt"])
        return [patches for _, _, patches in items]
    if op == "find":
        return [emtk.emtk_find_hits(ctx, items), state["out"]]
    if op == "infer":
        for adc, nticks, hits, scores in items:
            emtk.emtk_infer(ctx, adc, nticks, hits, scores)
    elif op == "batch":
        emtk.emtk_infer_batch(ctx, items)
    else:
        emtk.emtk_infer_batch_host(ctx, items)
    return [scores for _, _, _, scores in items]


def work(case):
    """Planes are counted as what their hits' windows can cover at most."""
    op, cols = case["op"], 8 if case["logits"] else 4
    if op == "patches":
        n = case["patches"]
        return {"bytes": n * (2304 * 4 + cols * 4) + W1_VALUES * W1_BYTES[case["precision"]], "flops": n * NET_FLOPS}
    shapes = _shapes(case)
    if op == "find":
        samples = sum(nw * case["nticks"] for nw, _, _ in shapes)
        return {"bytes": 4 * samples + 24 * len(shapes), "flops": samples}
    n = sum(nh for _, _, nh in shapes)
    planes = sum(min(nw * case["nticks"] * 4, nh * WINDOW_BYTES) for nw, _, nh in shapes)
    if op == "cut":
        return {"bytes": planes + n * (8 + 2304 * (4 if case["fmt"] == "f32" else 2)), "flops": planes // 4}
    calls = case["planes"] if op == "infer" else 1
    return {"bytes": planes + n * (8 + cols * 4) + calls * W1_VALUES * W1_BYTES[case["precision"]],
            "flops": n * NET_FLOPS}


def tolerance(case):
    if case["op"] == "cut":
        return "exact"  # the sum of the six ticks and its rounding are fixed
    if case["op"] == "find":
        return {"rel": 1e-6, "max": 1e-5, "differ": 0.0}  # the charge is a 32-bit sum
    # About four times what another order of the sums (other batches) or 64 bits showed: scores
    # at fp32 and tf32, scores and logits at the others.
    return {"fp32": {"rel": 4e-5, "max": 1e-3}, "tf32": {"rel": 1.2e-4, "max": 3e-3},
            "bf16": {"rel": 1e-2, "max": 0.1}, "fp16": {"rel": 2e-3, "max": 2e-2},
            "fp8": {"rel": 1e-2, "max": 0.1}}[case["precision"]]


# ------------------------------------------------------------- 64 bits
def _cut64(adc, hits, nticks):
    """Patches [n][48][48] in 64 bits: means of 6 ticks, zero outside the plane."""
    nw, nint = adc.shape[0], nticks // 6
    img = adc[:, :6 * nint].double().view(nw, nint, 6).sum(2) / 6
    img = torch.nn.functional.pad(img, (24, 24, 24, 24))
    span = torch.arange(48, device=DEV)
    w, b = hits[:, 0].long(), hits[:, 1].long().div(6, rounding_mode="floor")
    return img[(w[:, None] + span)[:, :, None], (b[:, None] + span)[:, None, :]]


def _net64(patches, wt, logits):
    out = []
    for p in patches.split(1024):
        x = p.double().unfold(1, 5, 1).unfold(2, 5, 1).reshape(-1, 25)  # [n * 1936][25], taps row by row
        x = torch.relu(x @ wt["conv_w"] + wt["conv_b"]).view(p.shape[0], -1)
        x = torch.relu(x @ wt["fc1_w"] + wt["fc1_b"])
        x = torch.relu(x @ wt["fc2_w"] + wt["fc2_b"])
        cls, mic = x @ wt["cls_w"] + wt["cls_b"], x @ wt["mic_w"] + wt["mic_b"]
        cols = [torch.softmax(cls, 1), torch.sigmoid(mic)]
        out.append(torch.cat(cols + ([cls, mic] if logits else []), 1))
    return torch.cat(out)


def _find64(adc, nticks, thr):
    """Maximal runs above thr: their number, hits (wire, first largest tick), extents, peak and sum."""
    x = adc[:, :nticks]
    above = x > thr
    before = torch.zeros_like(above)
    before[:, 1:] = above[:, :-1]
    w, t = above.nonzero(as_tuple=True)          # by wire, then tick
    v = x[above].double()
    run_of = (above & ~before)[above].long().cumsum(0) - 1
    n = int(run_of[-1]) + 1 if run_of.numel() else 0
    full = lambda fill, dt: torch.full((n,), fill, device=DEV, dtype=dt)
    peak = full(-math.inf, torch.float64).scatter_reduce(0, run_of, v, "amax")
    tick = torch.where(v == peak[run_of], t, nticks)
    at = full(nticks, torch.int64).scatter_reduce(0, run_of, tick, "amin")
    start = full(nticks, torch.int64).scatter_reduce(0, run_of, t, "amin")
    end = full(-1, torch.int64).scatter_reduce(0, run_of, t, "amax")
    wire = full(-1, torch.int64).scatter_reduce(0, run_of, w, "amax")
    charge = full(0.0, torch.float64).scatter_add(0, run_of, v)
    out = []
    room = adc.shape[0] * FIND_ROOM
    for cols in ([wire, at], [start, end], [peak, charge]):
        rows = torch.stack(cols, 1)[:room]
        out.append(torch.nn.functional.pad(rows, (0, 0, 0, room - rows.shape[0])))
    return n, [out[0].int(), out[1].int(), out[2]]


def exact(case, seed):
    data = _inputs(case, seed)
    op = case["op"]
    if op == "find":
        thr = torch.tensor(case["threshold"], dtype=torch.float32, device=DEV)
        found = [_find64(adc, case["nticks"], thr) for adc, _ in data]
        return [[n for n, _ in found], [torch.cat(cols) for cols in zip(*(rows for _, rows in found))]]
    if op == "cut":
        return [_cut64(adc, hits, case["nticks"]) for adc, hits in data]
    wt = {k: torch.from_numpy(v).to(DEV).double() for k, v in _weights().items()}
    wt["conv_w"] = wt["conv_w"].reshape(25, 48)
    if op == "patches":
        return _net64(data, wt, case["logits"])
    return [torch.cat([_net64(_cut64(adc, h, case["nticks"]), wt, case["logits"]) for h in hits.split(4096)])
            for adc, hits in data]
