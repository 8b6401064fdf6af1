"""GPU decode of calls whose frames are chained by prediction (Sec. III-D),
against the oracle: P runs that start and end inside a call and across calls,
more frames than a warp (32) and a CTA (256) of the mask kernel read at a
time, rows narrower and wider than the pixels a CTA sums (256) and than the
mask words it takes (32), every sample width, stage switches (no mask,
Zstandard mask) and several segments with single frames among them; small
calls, whose rows do it all, and ones large enough for the kernels around
them (8192 rows and 32 frames)."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2209_08196_gb300 import build as jbuild  # noqa: E402
from paper_2209_08196_gb300 import jiffy as J  # noqa: E402
from tests.gpu_util import TORCH_DT, to_np  # noqa: E402

jbuild.build()
DT = {1: np.uint8, 2: np.uint16, 4: np.uint32}


def runs_of_scans(rng, H, W, attrs, T):
    """Scans that mostly repeat the one before (P is chosen), now and then
    smooth ones unlike it (I is chosen), with zeros that come and go."""
    out, base = [], None
    for t in range(T):
        planes = []
        fresh = base is None or rng.random() < 0.12
        if fresh:
            smooth = rng.random() < 0.5
            base = []
            for s, _ in attrs:
                top = 1 << (8 * s)
                v = (np.arange(W)[None, :] // 7 + np.arange(H)[:, None] + rng.integers(1, 100)) % (top - 1) + 1 if smooth \
                    else rng.integers(1, top, size=(H, W), dtype=np.uint64)
                v = v.astype(np.int64)
                v[rng.random((H, W)) < 0.2] = 0
                base.append(v)
        for (s, _), b in zip(attrs, base):
            x = b + np.where(b > 0, rng.integers(-1, 2, size=b.shape), 0)
            x = np.clip(x, 0, (1 << (8 * s)) - 1)
            x[rng.random(x.shape) < 0.01] = 0
            planes.append(x.astype(DT[s]))
        out.append(planes)
    return out


CASES = [
    # H, W, attributes, frames per call, stages
    (3, 489, [(4, 10), (2, 1)], (40, 1, 2, 33), 0),
    (2, 1100, [(1, 1), (4, 1)], (3, 66), 0),
    (1, 31, [(2, 3)], (70,), 0),
    (2, 2049, [(2, 1)], (5, 4), 0),
    (4, 256, [(1, 1)], (34, 2), J.STAGE_NO_MASK),
    (3, 300, [(2, 1), (1, 1)], (35, 2), J.STAGE_ZSTD_MASK),
    (3, 512, [(4, 1)], (33, 3), J.STAGE_ZSTD_MASK),
    (2, 520, [(2, 1)], (6, 3), J.STAGE_NO_DELTA),
    # (the first or only call of these is a large one)
    (128, 40, [(2, 1), (1, 1)], (33, 3), 0),
    (64, 601, [(4, 10), (1, 1)], (70, 2), 0),
    (32, 1100, [(4, 1)], (290,), 0),
    (128, 300, [(2, 1), (1, 1)], (33, 2), J.STAGE_ZSTD_MASK),
    (128, 65, [(2, 1)], (65,), J.STAGE_NO_MASK),
]


@pytest.mark.parametrize("H,W,attrs,calls,stages", CASES)
def test_predicted_frames_match_the_oracle(H, W, attrs, calls, stages):
    rng = np.random.default_rng(H * 10007 + W)
    ref, refd = oracle.Codec(H, W, attrs, stages=stages), oracle.Codec(H, W, attrs, stages=stages)
    dec = J.jiffy_stream_create(J.JIFFY_DECODER, H, W, attrs, stages=stages)
    scans = runs_of_scans(rng, H, W, attrs, sum(calls))
    seen, at = set(), 0
    for T in calls:
        parts = [ref.encode(s, return_modes=True) for s in scans[at:at + T]]
        at += T
        seen |= {m for _, modes in parts for m in modes}
        frames = [b for b, _ in parts]
        # the stream header, if any, belongs to the first frame's bytes
        first = 16 + 8 * len(attrs) if at == T else 0
        ends = np.cumsum([len(f) for f in frames]).tolist()
        buf = torch.from_numpy(np.frombuffer(b"".join(frames), dtype=np.uint8).copy()).cuda()
        planes = [torch.zeros((T, H, W), dtype=TORCH_DT[s], device="cuda") for s, _ in attrs]
        J.jiffy_decode_seq(dec, buf, buf.numel(), [first] + ends, planes)
        for t, f in enumerate(frames):
            want, _ = refd.decode(f)
            for k, (s, _) in enumerate(attrs):
                assert np.array_equal(to_np(planes[k][t], s), want[k]), (at - T + t, k)
    assert 1 in seen and (0 in seen)


SMALL = [(2, 97, [(1, 1)], 1), (3, 600, [(4, 10), (1, 1)], 9), (1, 64, [(2, 1)], 1), (2, 3000, [(2, 1)], 4), (5, 40, [(4, 1)], 1)]


@pytest.mark.parametrize("sensors", [SMALL, SMALL + [(120, 50, [(1, 1), (4, 1)], 36)], [(64, 77, [(2, 1)], 5)] * 260 + [(1, 33, [(1, 1)], 32)]])
def test_batch_of_single_and_several_frames(sensors):
    rng = np.random.default_rng(5)
    decs, bufs, offs, lens, planes, wants = [], [], [], [], [], []
    for H, W, attrs, T in sensors:
        ref, refd = oracle.Codec(H, W, attrs), oracle.Codec(H, W, attrs)
        frames = [ref.encode(s) for s in runs_of_scans(rng, H, W, attrs, T)]
        wants.append([refd.decode(f)[0] for f in frames])
        bufs.append(torch.from_numpy(np.frombuffer(b"".join(frames), dtype=np.uint8).copy()).cuda())
        offs.append([16 + 8 * len(attrs)] + np.cumsum([len(f) for f in frames]).tolist())
        lens.append(offs[-1][-1])
        planes.append([torch.zeros((T, H, W), dtype=TORCH_DT[s], device="cuda") for s, _ in attrs])
        decs.append(J.jiffy_stream_create(J.JIFFY_DECODER, H, W, attrs))
    J.jiffy_decode_batch(J.jiffy_batch_create(), decs, bufs, lens, offs, planes)
    for (H, W, attrs, T), got, want in zip(sensors, planes, wants):
        for t in range(T):
            for k, (s, _) in enumerate(attrs):
                assert np.array_equal(to_np(got[k][t], s), want[t][k]), (H, W, t, k)


# Calls large enough for the kernels around the rows, whose state nothing but
# those kernels clears when they are enqueue-only, and malformed ones among
# them. Runs of two P frames are added by rows that wait, long ones behind the
# rows (3000 rows per frame of the longest run).
BIG = (128, 65, [(2, 1), (1, 1)])
ZERO_ROW = 7  # a row without samples: its chunk is one class word


def predicted(rng, T, run):
    """Frames of noise, each followed by `run` near copies of it (coded P)."""
    H, W, attrs = BIG
    out = []
    for t in range(T):
        if t % (run + 1) == 0:
            base = [rng.integers(1, 1 << (8 * s), size=(H, W)) for s, _ in attrs]
        planes = []
        for (s, _), b in zip(attrs, base):
            x = np.clip(b + rng.integers(-1, 2, size=b.shape), 1, (1 << (8 * s)) - 1)
            x[rng.random(x.shape) < 0.1] = 0
            x[ZERO_ROW] = 0
            planes.append(x.astype(DT[s]))
        out.append(planes)
    return out


def coded(ref, refd, scans, waits):
    """(stream bytes, frame offsets, planes) of a call's scans by the oracle;
    waits: whether the rows of its P runs wait for one another."""
    H, W, attrs = BIG
    parts = [ref.encode(s, return_modes=True) for s in scans]
    longest = 0
    for a in range(len(attrs)):
        run = 0
        for t, (_, modes) in enumerate(parts):
            run = run + 1 if t and modes[a] == 1 else 0
            longest = max(longest, run)
    rows = len(scans) * len(attrs) * H
    assert len(scans) >= 32 and rows >= 8192 and longest >= 2
    assert (longest * 3000 <= rows) == waits, longest
    ends = np.cumsum([len(b) for b, _ in parts]).tolist()
    return b"".join(b for b, _ in parts), ends, [refd.decode(b)[0] for b, _ in parts]


def on_gpu(data):
    return torch.from_numpy(np.frombuffer(bytes(data), dtype=np.uint8).copy()).cuda()


def check_planes(planes, want, what=""):
    for t, w in enumerate(want):
        for k, (s, _) in enumerate(BIG[2]):
            assert np.array_equal(to_np(planes[k][t], s), w[k]), (what, t, k)


def test_enqueued_calls_clear_what_the_calls_before_them_left():
    # four enqueue-only calls in flight on one handle before the wait, the
    # P runs of some summed and of some waited for, then all of them again
    H, W, attrs = BIG
    rng = np.random.default_rng(41)
    ref, refd = oracle.Codec(H, W, attrs), oracle.Codec(H, W, attrs)
    dec = J.jiffy_stream_create(J.JIFFY_DECODER, H, W, attrs)
    calls = []
    for i, (T, run) in enumerate(((40, 1000), (33, 2), (40, 2), (64, 1000))):
        data, ends, want = coded(ref, refd, predicted(rng, T, run), run == 2)
        offs = torch.tensor([16 + 8 * len(attrs) if i == 0 else 0] + ends, dtype=torch.int64, device="cuda")
        calls.append((on_gpu(data), offs, want))
    for _ in range(2):
        J.jiffy_stream_reset(dec)
        outs = []
        for src, offs, want in calls:
            outs.append([torch.zeros((len(want), H, W), dtype=TORCH_DT[s], device="cuda") for s, _ in attrs])
            J.jiffy_decode_seq_async(dec, src, offs, outs[-1])
        J.jiffy_stream_wait(dec)
        for i, ((_, _, want), planes) in enumerate(zip(calls, outs)):
            check_planes(planes, want, i)


def damaged(data, ends, kind, t):
    """The stream with frame t of its call damaged (attribute 0)."""
    H, W, attrs = BIG
    b = bytearray(data)
    f = ends[t - 1]                          # frame t's header
    sec = f + 8 + 12 * len(attrs)            # its first section: the row table
    end = lambda r: int.from_bytes(b[sec + 8 * r:sec + 8 * r + 4], "little")  # noqa: E731
    chunk = lambda r: sec + 8 * H + (end(r - 1) if r else 0)  # noqa: E731
    if kind == "mode":
        b[f + 8] = 2
    elif kind == "section bytes":
        b[f + 12] ^= 4
    elif kind == "row end":
        b[sec + 8 * 5] ^= 8
    elif kind == "row end far away":
        b[sec + 8 * 5:sec + 8 * 5 + 4] = (0xFFFFFFF0).to_bytes(4, "little")
    elif kind == "invalid class":
        b[chunk(5)] = 0xFF
    elif kind == "literals for every word":
        b[chunk(5)] = 0x2A
    elif kind == "literals past the chunk":
        assert end(ZERO_ROW) - end(ZERO_ROW - 1) == 4
        b[chunk(ZERO_ROW)] = 0x2A
    else:  # a block of 40 bits
        cls = b[chunk(5)]
        lits = sum((cls >> (2 * j)) & 3 == 2 for j in range(3))
        b[chunk(5) + 4 * (1 + lits)] = 40
    return b


KINDS = ["mode", "section bytes", "row end", "row end far away", "invalid class", "literals for every word",
         "literals past the chunk", "block width"]


@pytest.mark.parametrize("run", [2, 1000])
@pytest.mark.parametrize("kind", KINDS)
def test_damaged_frames_inside_a_run_are_refused(kind, run):
    # in a P frame, and in an I or P frame whose successor is coded P; the
    # decoder goes on with the undamaged stream, blocking and enqueue-only
    H, W, attrs = BIG
    T = 40
    rng = np.random.default_rng(run)
    data, ends, want = coded(oracle.Codec(H, W, attrs), oracle.Codec(H, W, attrs), predicted(rng, T, run), run == 2)
    offs = [16 + 8 * len(attrs)] + ends
    d_offs = torch.tensor(offs, dtype=torch.int64, device="cuda")
    dec = J.jiffy_stream_create(J.JIFFY_DECODER, H, W, attrs)
    good = on_gpu(data)
    for t in (6, 7):
        b = damaged(data, ends, kind, t)
        refd = oracle.Codec(H, W, attrs)
        with pytest.raises(oracle.OracleError):
            for k in range(t + 1):
                refd.decode(bytes(b[(ends[k - 1] if k else 0):ends[k]]))
        bad = on_gpu(b)
        planes = [torch.zeros((T, H, W), dtype=TORCH_DT[s], device="cuda") for s, _ in attrs]
        J.jiffy_stream_reset(dec)
        with pytest.raises(J.JiffyError) as ei:
            J.jiffy_decode_seq(dec, bad, bad.numel(), offs, planes)
        assert ei.value.name == "JIFFY_ERR_CORRUPT"
        assert J.jiffy_stream_frame_index(dec) == 0
        J.jiffy_decode_seq(dec, good, good.numel(), offs, planes)
        check_planes(planes, want, "blocking")
        planes = [torch.zeros_like(p) for p in planes]
        J.jiffy_stream_reset(dec)
        J.jiffy_decode_seq_async(dec, bad, d_offs, planes)
        with pytest.raises(J.JiffyError) as ei:
            J.jiffy_stream_wait(dec)
        assert ei.value.name == "JIFFY_ERR_CORRUPT"
        J.jiffy_stream_reset(dec)
        J.jiffy_decode_seq_async(dec, good, d_offs, planes)
        J.jiffy_stream_wait(dec)
        check_planes(planes, want, "enqueue-only")


@pytest.mark.parametrize("run", [2, 1000])
def test_bounded_wait_of_a_large_call_runs_out_and_the_stream_recovers(run):
    # one row withholds its completion flag (host-side hook; the rows of every
    # P run then wait): the same row of the next frame gives up after the
    # bounded wait, the rest of the call goes on, the stream's state is as
    # before and the same frames decode next
    H, W, attrs = BIG
    T = 40
    rng = np.random.default_rng(100 + run)
    data, ends, want = coded(oracle.Codec(H, W, attrs), oracle.Codec(H, W, attrs), predicted(rng, T, run), run == 2)
    src, offs = on_gpu(data), [16 + 8 * len(attrs)] + ends
    planes = [torch.zeros((T, H, W), dtype=TORCH_DT[s], device="cuda") for s, _ in attrs]
    dec = J.jiffy_stream_create(J.JIFFY_DECODER, H, W, attrs)
    J.jiffy_stream_test_withhold_row(dec, 3 * H + 5)  # attribute 0, scan 3 (scan 4 is coded P), row 5
    with pytest.raises(J.JiffyError) as ei:
        J.jiffy_decode_seq(dec, src, len(data), offs, planes)
    assert ei.value.name == "JIFFY_ERR_TIMEOUT"
    assert J.jiffy_stream_frame_index(dec) == 0
    J.jiffy_decode_seq(dec, src, len(data), offs, planes)
    check_planes(planes, want)
