"""Encoder packing at every block width (Sec. II, PFOR) against the oracle: the
low bits are assembled four, two or one values at a time as the widths of a
1024-value step allow (8 and 16 bits), with and without exceptions, blocks and
steps ending anywhere, with the delta stage's fast and general forms (deltas of
2^30 and more) and without it."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2209_08196_gb300 import build as jbuild  # noqa: E402
from paper_2209_08196_gb300 import jiffy as J  # noqa: E402
from tests.gpu_util import GpuCodec  # noqa: E402

jbuild.build()


@pytest.mark.parametrize("stages", [0, J.STAGE_NO_DELTA, J.STAGE_NO_DELTA | J.STAGE_NO_ZIGZAG | J.STAGE_NO_MASK])
@pytest.mark.parametrize("bits", [1, 6, 7, 8, 9, 14, 15, 16, 17, 28, 29, 30, 31, 32])
def test_every_packing_width(bits, stages):
    rng = np.random.default_rng(bits)
    W = 1024 + 128 + 37
    rows = []
    for share in (0.0, 0.0, 0.02, 0.2):  # values wider than most
        v = rng.integers(0, 1 << bits, W, dtype=np.uint64) if bits < 32 else rng.integers(0, 1 << 32, W, dtype=np.uint64)
        wide = rng.random(W) < share
        v[wide] = rng.integers(0, 1 << min(32, bits + 9), int(wide.sum()), dtype=np.uint64)
        v[rng.random(W) < 0.05] = 0
        rows.append(v)
    for at in (5, 600, 1100):  # blocks of another width in the same step
        rows[1][at:at + 80] = rng.integers(1, 4, 80)
    scan = [np.stack(rows).astype(np.uint32)]
    attrs = [(4, 1)]
    got = GpuCodec(len(rows), W, attrs, force_mode=0, stages=stages).encode(scan)
    assert got == oracle.encode_sequence(len(rows), W, attrs, [scan], force_mode=0, stages=stages)[0]
