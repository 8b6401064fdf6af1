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
