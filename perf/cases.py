"""The work that programs built on this codec have it do, as cases to be timed.

A case is a dict of plain values. `prepare` makes what a user's program holds before the call (scans on the GPU, stream
or batch handles, output buffers, for a decode the recorded stream), `run` makes one pass through the public entry
points of paper_2209_08196_gb300.jiffy and returns what the pass wrote: stream bytes and frame offsets, decoded planes,
or range and attribute images. Everything the codec does is integer work, so every output is exact.

Scans come from the ray-cast scenes of paper_2209_08196_gb300.synth (a spinning sensor among boxes on a ground plane),
with the noise and dropouts drawn on the GPU:
  open    driving, sky and far returns missing, 8 % dropouts
  drive   driving inside an enclosing wall, 12 % dropouts (the benchmark's scene)
  parked  sensor at rest, dropouts mostly on the same pixels, 10 mm range noise (P scans are chosen for the ranges)
  walk    random yaw and translation, zeros in discs of 5 to 40 pixels (I scans are chosen)
"""
import math
import random

import torch

from paper_2209_08196_gb300 import jiffy as J
from paper_2209_08196_gb300 import synth

ATTRS = {
    "range": (synth.RANGE,),
    "range+signal": (synth.RANGE, synth.SIGNAL),
    "range+reflectivity": (synth.RANGE, synth.REFLECTIVITY),
    "all": (synth.RANGE, synth.RANGE2, synth.SIGNAL, synth.REFLECTIVITY, synth.AMBIENT),
}
# raw bytes per stream byte, about, by scene (for work(): a stream's size is only known once it is coded)
RATIO = {"open": 8.0, "drive": 4.4, "parked": 4.0, "walk": 7.2}
LIVE_SCANS = 8  # scans that a live case goes through, one per pass, before it starts again
MAX_RAW = 540 << 20  # raw bytes of the largest listed case, the bound of the drawn ones


def _case(name, kind, op, call, scene, H, W, attrs, T, prec=10, zstd=False):
    return {"name": name, "kind": kind, "op": op, "call": call, "scene": scene, "H": H, "W": W, "attrs": attrs, "T": T,
            "prec": prec, "zstd": zstd}


def _fleet_case(name, op, scene, sensors, mix, graphs):
    """One batched call over `sensors` streams; their shapes, attribute sets and scan counts follow from `mix`."""
    return {"name": name, "kind": "batch", "op": op, "scene": scene, "sensors": sensors, "mix": mix, "graphs": graphs}


def listed():
    return [
        # a live sensor's scan coded as it arrives, one blocking call per scan: latency
        _case("live_encode_64x1024", "stream", "encode", "scan", "open", 64, 1024, "range", 1),
        # the receiving side of that link
        _case("live_decode_64x1024", "stream", "decode", "scan", "open", 64, 1024, "range", 1),
        # a recording of a 128-beam sensor with all its attributes, ten seconds per enqueue-only call
        _case("record_encode_100x128x2048", "stream", "encode", "async", "drive", 128, 2048, "all", 100),
        # the replay of that recording
        _case("replay_decode_100x128x2048", "stream", "decode", "async", "drive", 128, 2048, "all", 100),
        # a roadside sensor cropped to the window that it watches: rows of an odd width, the ranges predicted from scan to scan
        _case("parked_encode_100x64x489", "stream", "encode", "seq", "parked", 64, 489, "range+signal", 100),
        _case("parked_decode_100x64x489", "stream", "decode", "seq", "parked", 64, 489, "range+signal", 100),
        # a mapping walk archived in one go at 1 mm, and read back: the largest calls
        _case("walk_encode_410x128x2048", "stream", "encode", "seq", "walk", 128, 2048, "range+reflectivity", 410, prec=1),
        _case("walk_decode_410x128x2048", "stream", "decode", "seq", "walk", 128, 2048, "range+reflectivity", 410, prec=1),
        # a server coding what 64 sensors of several kinds have queued, in one batched call each way
        _fleet_case("fleet_encode_64", "encode", "drive", 64, 7, True),
        _fleet_case("fleet_decode_64", "decode", "drive", 64, 7, True),
        # the stream option that codes the masks as Zstandard frames, written and read back
        _case("zstd_roundtrip_40x128x2048", "stream", "roundtrip", "async", "drive", 128, 2048, "all", 40, zstd=True),
        # the step before the codec: point clouds to range and attribute images
        _case("points_40x128x2048", "points", "standardize", "seq", "drive", 128, 2048, "all", 40),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["scan", "async", "async", "seq", "seq", "batch", "zstd", "points"])
    if kind == "batch":
        return _unnamed(_fleet_case("", rng.choice(["encode", "decode"]), rng.choice(["drive", "parked"]),
                                    _log_int(rng, 2, 48), rng.randrange(1 << 20), rng.random() < 0.5))
    H = _log_int(rng, 8, 128)
    W = _log_int(rng, 256, 4096)
    if rng.random() < 0.5:  # sensors' own widths are multiples of 64; cropped ones are anything
        W = max(256, W // 64 * 64)
    attrs = rng.choice(sorted(ATTRS))
    scene = rng.choice(sorted(RATIO))
    raw = H * W * sum(synth.ATTR_DTYPE[a] for a in ATTRS[attrs])
    most = max(1, min(410, (MAX_RAW // (4 if kind in ("zstd", "points") else 1)) // raw))
    most = min(most, 200 if kind == "points" else 100 if scene == "parked" else 410)  # (predicted frames depend on one another)
    T = 1 if kind == "scan" else min(most, _log_int(rng, 2, 410))
    prec = rng.choice([1, 2, 3, 5, 10, 10, 16, 50])
    if kind == "points":
        return _unnamed(_case("", "points", "standardize", "seq", rng.choice(["drive", "walk"]), H, W, attrs, T))
    op = rng.choice(["encode", "decode"])
    if kind == "zstd":
        return _unnamed(_case("", "stream", op, rng.choice(["async", "seq"]), scene, H, W, attrs, T, prec, zstd=True))
    return _unnamed(_case("", "stream", op, kind, scene, H, W, attrs, T, prec))


def _unnamed(c):
    return {k: v for k, v in c.items() if k != "name"}


# ---------------------------------------------------------------- inputs
def _descs(attrs, prec):
    return [(synth.ATTR_DTYPE[a], prec if a in (synth.RANGE, synth.RANGE2) else 1) for a in attrs]


def _discs(gen, H, W, frac):
    """Zeros in discs of radius 5 to 40 pixels covering about `frac` of the image (H x W truth values)."""
    n = max(1, round(-math.log(1.0 - frac) * (H + 40) * (W + 40) / 1860.0))  # 1860: a disc's mean area
    u = torch.rand((3, n), generator=gen, device="cuda")
    cy, cx, rad = u[0] * (H + 40) - 20, u[1] * (W + 40) - 20, 5.0 + 35.0 * u[2]
    y = torch.arange(H, device="cuda", dtype=torch.float32)
    x = torch.arange(W, device="cuda", dtype=torch.float32)
    dy = (y[None] - cy[:, None]) ** 2
    half = (rad[:, None] ** 2 - dy).clamp_min(0).sqrt()  # half chord of each disc on each row
    inside = dy <= rad[:, None] ** 2
    # chords as +1 / -1 at their ends, summed along the row
    lo = (cx[:, None] - half).ceil().clamp(0, W).long()
    hi = ((cx[:, None] + half).floor() + 1).clamp(0, W).long()
    ends = torch.zeros((H, W + 1), dtype=torch.int32, device="cuda")
    rows = torch.arange(H, device="cuda")[None].expand(n, H)
    one = inside.int()
    ends.index_put_((rows, lo), one, accumulate=True)
    ends.index_put_((rows, hi), -one, accumulate=True)
    return ends.cumsum(1)[:, :W] > 0


def _scans(scene, attrs, H, W, T, seed):
    """[T x H x W tensor per attribute] of seeded scans, in the containers that the codec takes."""
    walk = scene == "walk"
    cfg = synth.SensorConfig(H=H, W=W, attrs=attrs, n_scans=T, wall=scene != "open", seed=seed, random_motion=walk,
                             yaw_rate_dps=30.0 if walk else 0.0,
                             speed_mps=0.0 if scene == "parked" else 3.0 if walk else 10.0)
    seq = synth.ScanSequence(cfg, device="cuda")
    gen = torch.Generator(device="cuda").manual_seed(seed * 1000003 + 11)

    def rand():
        return torch.rand((H, W), generator=gen, device="cuda")

    def randn():
        return torch.randn((H, W), generator=gen, device="cuda")

    dead = rand()
    out = [torch.empty((T, H, W), dtype=J.TORCH_DTYPE[synth.ATTR_DTYPE[a]], device="cuda") for a in attrs]
    rows = torch.arange(H, device="cuda", dtype=torch.float32)[:, None] / H
    cols = torch.arange(W, device="cuda", dtype=torch.float32)[None, :] / W
    field = 1500.0 + sum(float(seq.amb_amp[k]) * torch.sin(2 * math.pi * (float(seq.amb_k[k, 0]) * rows + float(
        seq.amb_k[k, 1]) * cols) + float(seq.amb_phase[k])) for k in range(4))
    hit = None
    for t in range(T):
        if hit is None or scene != "parked":
            hit = seq._cast(t)
        near, second, refl = hit
        valid = near <= synth.MAX_RANGE_M
        if walk:
            valid = valid & ~_discs(gen, H, W, 0.4)
        elif scene == "parked":
            valid = valid & (dead >= 0.108) & (rand() >= 0.012)
        else:
            valid = valid & (rand() >= (0.08 if scene == "open" else 0.12))
        zero = torch.zeros_like(near)
        for plane, a in zip(out, attrs):
            if a == synth.RANGE:
                r = near + randn() * 0.01 if scene == "parked" else near
                v = torch.where(valid, (r * 1000.0).round().clamp_min(1.0), zero)
            elif a == synth.RANGE2:  # a second return at depth edges
                edge = torch.zeros_like(valid)
                jump = (near[:, 1:] - near[:, :-1]).abs() > 0.5
                edge[:, 1:] |= jump
                edge[:, :-1] |= jump
                v = torch.where(valid & edge & (second <= synth.MAX_RANGE_M), (second * 1000.0).round(), zero)
            elif a == synth.SIGNAL:
                lam = (1000.0 * refl / near.clamp(1.0, 1e4) ** 2).clamp(0, 60000)
                v = torch.where(valid, torch.poisson(lam, generator=gen).clamp(1, 65535), zero)
            elif a == synth.REFLECTIVITY:
                v = torch.where(valid, (refl + (rand() * 7).floor() - 3).clamp(1, 255), zero)
            else:
                v = (field + randn() * 20.0).round().clamp(1, 65535)
            v = v.to(torch.int32)
            plane[t] = torch.where(v >= 1 << 15, v - (1 << 16), v).to(torch.int16) if plane.dtype == torch.int16 else v.to(plane.dtype)
    return out


def _fleet(case):
    """[(H, W, attributes, scans queued)] of a batched case's sensors: the many-stream shapes and attribute sets."""
    r = random.Random(case["mix"])
    return [(*r.choice(synth.BATCH_SHAPES), r.choice(synth.BATCH_ATTR_SETS), r.randint(1, 8)) for _ in range(case["sensors"])]


def _points(case, seed):
    """The valid pixels of each scan as points (metres, in the scans' row-major order), with float attribute values."""
    H, W, T = case["H"], case["W"], case["T"]
    names = [a for a in ATTRS[case["attrs"]] if a not in (synth.RANGE, synth.RANGE2)]
    scans = _scans(case["scene"], (synth.RANGE, *names), H, W, T, seed)
    gen = torch.Generator(device="cuda").manual_seed(seed * 1000003 + 29)
    el = torch.deg2rad(torch.linspace(22.5, -22.5, H, device="cuda", dtype=torch.float64))
    spacing = math.radians(45.0 / max(1, H - 1))
    xyz, values, offsets = [], [[] for _ in names], [0]
    for t in range(T):
        rng_mm = scans[0][t]
        at = (rng_mm > 0).nonzero()
        y, x = at[:, 0], at[:, 1]
        d = rng_mm[y, x].double() / 1000.0
        jitter = torch.rand((2, len(d)), generator=gen, device="cuda", dtype=torch.float64) * 0.6 - 0.3
        az = (x + 0.5 + jitter[0]) * (2 * math.pi / W)
        e = el[y] + jitter[1] * spacing
        xyz.append(torch.stack([d * e.cos() * az.cos(), d * e.cos() * az.sin(), d * e.sin()], 1).float())
        for v, plane in zip(values, scans[1:]):
            v.append(plane[t][y, x].float())
        offsets.append(offsets[-1] + len(d))
    return torch.cat(xyz).contiguous(), [torch.cat(v) for v in values], offsets, [scans[1 + i].dtype for i in range(len(names))]


# ---------------------------------------------------------------- a user's program
def _zeros(n):
    return torch.zeros(n, dtype=torch.uint8, device="cuda")


def prepare(case, seed):
    if case["kind"] == "batch":
        return _prepare_batch(case, seed)
    if case["kind"] == "points":
        H, W, T = case["H"], case["W"], case["T"]
        xyz, values, offsets, types = _points(case, seed)
        sensor = J.jiffy_standardizer_create(H, W, [math.radians(22.5 - 45.0 * r / max(1, H - 1)) for r in range(H)])
        images = [torch.zeros((T, H, W), dtype=t, device="cuda") for t in [torch.int32] + types]
        return {"case": case, "sensor": sensor, "xyz": xyz, "offsets": offsets, "range": images[0],
                "attrs": [(v, o, 1.0) for v, o in zip(values, images[1:])]}
    attrs, H, W = ATTRS[case["attrs"]], case["H"], case["W"]
    live = case["call"] == "scan"
    T = LIVE_SCANS if live else case["T"]
    planes = _scans(case["scene"], attrs, H, W, T, seed)
    desc = _descs(attrs, case["prec"])
    stages = J.STAGE_ZSTD_MASK if case["zstd"] else 0
    enc = J.jiffy_stream_create(J.JIFFY_ENCODER, H, W, desc, stages=stages)
    st = {"case": case, "T": T, "next": 0}
    if live:
        scans = [[p[t] for p in planes] for t in range(T)]
        if case["op"] == "encode":
            return {**st, "enc": enc, "scans": scans, "out": _zeros(J.jiffy_max_encoded_size(H, W, desc))}
        dec = J.jiffy_stream_create(J.JIFFY_DECODER, H, W, desc, stages=stages)
        frames = []
        for s in scans:
            out = _zeros(J.jiffy_max_encoded_size(H, W, desc))
            frames.append(out[: J.jiffy_encode(enc, s, out)].clone())
        return {**st, "dec": dec, "frames": frames, "planes": J.empty_planes(dec)}
    if case["op"] == "encode":
        # room for a recording that does not shrink; what a pass leaves unwritten stays zero
        room = sum(p.numel() * p.element_size() for p in planes) + 8 * H * T * len(attrs) + 4096
        return {**st, "enc": enc, "scans": planes, "out": _zeros(min(room, J.jiffy_max_encoded_size(H, W, desc, T))),
                "offsets": torch.zeros(T + 1, dtype=torch.int64, device="cuda")}
    dec = J.jiffy_stream_create(J.JIFFY_DECODER, H, W, desc, stages=stages)
    out = _zeros(J.jiffy_max_encoded_size(H, W, desc, T))
    st.update(dec=dec, planes=[p.zero_() for p in J.empty_planes(dec, T)])
    if case["op"] == "roundtrip":
        return {**st, "enc": enc, "scans": planes, "out": out, "offsets": torch.zeros(T + 1, dtype=torch.int64, device="cuda")}
    n, offsets = J.jiffy_encode_seq(enc, planes, out)
    stream = out[:n].clone()
    return {**st, "stream": stream, "host_offsets": offsets, "offsets": torch.tensor(offsets, dtype=torch.int64, device="cuda")}


def _arena(sizes):
    """One zeroed buffer with room for each size, and its parts, each on a 256-byte boundary."""
    at, starts = 0, []
    for n in sizes:
        starts.append(at)
        at += -(-n // 256) * 256
    buf = _zeros(max(at, 256))
    return buf, [buf[a:a + n] for a, n in zip(starts, sizes)]


def _prepare_batch(case, seed):
    batch = J.jiffy_batch_create()
    if case["graphs"]:
        J.jiffy_batch_set_graphs(batch, True)
    fleet = [(H, W, attrs, T, _descs(attrs, 10)) for H, W, attrs, T in _fleet(case)]
    scans = [_scans(case["scene"], attrs, H, W, T, seed * 4099 + i) for i, (H, W, attrs, T, _) in enumerate(fleet)]
    enc = [J.jiffy_stream_create(J.JIFFY_ENCODER, H, W, desc) for H, W, _, _, desc in fleet]
    buf, outs = _arena([J.jiffy_max_encoded_size(H, W, desc, T) for H, W, _, T, desc in fleet])
    if case["op"] == "encode":
        return {"case": case, "batch": batch, "enc": enc, "scans": scans, "buffer": buf, "outs": outs}
    coded = J.jiffy_encode_batch(J.jiffy_batch_create(), enc, scans, outs)
    images, parts = _arena([p.numel() * p.element_size() for s in scans for p in s])
    parts = iter(parts)
    planes = [[next(parts).view(p.dtype).view(p.shape) for p in s] for s in scans]
    return {"case": case, "batch": batch, "dec": [J.jiffy_stream_create(J.JIFFY_DECODER, H, W, desc) for H, W, _, _, desc in fleet],
            "streams": [o[:n].clone() for o, (n, _) in zip(outs, coded)], "lengths": [n for n, _ in coded],
            "host_offsets": [f for _, f in coded], "buffer": images, "planes": planes}


def run(state):
    case = state["case"]
    if case["kind"] == "points":
        J.jiffy_standardize_seq(state["sensor"], state["xyz"], state["offsets"], state["range"], state["attrs"])
        return {"range": state["range"], "attrs": [o for _, o, _ in state["attrs"]]}
    if case["kind"] == "batch":
        return _run_batch(state)
    if case["call"] == "scan":  # the stream goes on from pass to pass
        i, state["next"] = state["next"], (state["next"] + 1) % state["T"]
        if case["op"] == "encode":
            n = J.jiffy_encode(state["enc"], state["scans"][i], state["out"])
            return {"stream": state["out"], "bytes": n}
        if i == 0:
            J.jiffy_stream_reset(state["dec"])
        J.jiffy_decode(state["dec"], state["frames"][i], state["frames"][i].numel(), state["planes"])
        return {"planes": state["planes"]}
    if case["op"] in ("encode", "roundtrip"):  # each call starts a recording of its own
        J.jiffy_stream_reset(state["enc"])
        if case["call"] == "seq":
            n, offsets = J.jiffy_encode_seq(state["enc"], state["scans"], state["out"])
            return {"stream": state["out"], "bytes": n, "offsets": torch.tensor(offsets)}
        J.jiffy_encode_seq_async(state["enc"], state["scans"], state["out"], state["offsets"])
        if case["op"] == "encode":
            return {"stream": state["out"], "offsets": state["offsets"]}
    J.jiffy_stream_reset(state["dec"])
    if case["op"] == "roundtrip":
        J.jiffy_decode_seq_async(state["dec"], state["out"], state["offsets"], state["planes"])
        return {"stream": state["out"], "offsets": state["offsets"], "planes": state["planes"]}
    if case["call"] == "seq":
        J.jiffy_decode_seq(state["dec"], state["stream"], state["stream"].numel(), state["host_offsets"], state["planes"])
    else:
        J.jiffy_decode_seq_async(state["dec"], state["stream"], state["offsets"], state["planes"])
    return {"planes": state["planes"]}


def _run_batch(state):
    if state["case"]["op"] == "encode":
        for h in state["enc"]:
            J.jiffy_stream_reset(h)
        coded = J.jiffy_encode_batch(state["batch"], state["enc"], state["scans"], state["outs"])
        return {"offsets": torch.tensor([x for _, f in coded for x in f]), "streams": state["buffer"]}
    for h in state["dec"]:
        J.jiffy_stream_reset(h)
    J.jiffy_decode_batch(state["batch"], state["dec"], state["streams"], state["lengths"], state["host_offsets"], state["planes"])
    return {"planes": state["buffer"]}


# ---------------------------------------------------------------- what a pass cannot do without
def work(case):
    if case["kind"] == "batch":
        raw = sum(H * W * T * sum(synth.ATTR_DTYPE[a] for a in attrs) for H, W, attrs, T in _fleet(case))
        return {"bytes": raw + raw / RATIO[case["scene"]], "flops": 0}
    px = case["H"] * case["W"] * case["T"]
    names = ATTRS[case["attrs"]]
    if case["kind"] == "points":  # about 12 (40 in discs) % of the pixels have no point; points in, images out
        extra = [a for a in names if a not in (synth.RANGE, synth.RANGE2)]
        full = 0.6 if case["scene"] == "walk" else 0.88
        return {"bytes": px * full * (12 + 4 * len(extra)) + px * (4 + sum(synth.ATTR_DTYPE[a] for a in extra)), "flops": 0}
    raw = px * sum(synth.ATTR_DTYPE[a] for a in names)
    once = raw + raw / RATIO[case["scene"]]
    return {"bytes": once * (2 if case["op"] == "roundtrip" else 1), "flops": 0}


def tolerance(case):
    return "exact"  # integers and bytes throughout
