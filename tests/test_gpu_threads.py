"""GPU: streams used by several host threads at once are independent, also when
their rows differ in width (the rows kernels' shared memory is sized by the
widest row of a call, the kernels themselves are shared by all threads)."""
import threading

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2209_08196_gb300 import build as jbuild  # noqa: E402
from paper_2209_08196_gb300 import jiffy as J  # noqa: E402
from tests.gpu_util import to_dev  # noqa: E402

jbuild.build()


@pytest.mark.parametrize("H,T", [(4, 2), (256, 33)])  # one kernel to decode; the kernels around the rows as well
def test_streams_of_several_threads_and_widths(H, T):
    attrs = [(2, 1)]
    errors = []
    start = threading.Barrier(4)

    def work(W):
        try:
            v = np.random.default_rng(W).integers(0, 900, size=(T, H, W)).astype(np.uint16)
            planes = to_dev(v)
            enc = J.jiffy_stream_create(J.JIFFY_ENCODER, H, W, attrs)
            dec = J.jiffy_stream_create(J.JIFFY_DECODER, H, W, attrs)
            out = torch.zeros(J.jiffy_max_encoded_size(H, W, attrs, T), dtype=torch.uint8, device="cuda")
            stream = torch.cuda.Stream()
            torch.cuda.synchronize()
            start.wait()
            for _ in range(150):
                J.jiffy_stream_reset(enc)
                J.jiffy_stream_reset(dec)
                got = torch.zeros_like(planes)
                torch.cuda.current_stream().synchronize()
                n, offs = J.jiffy_encode_seq(enc, [planes], out, stream)
                J.jiffy_decode_seq(dec, out, n, offs, [got], stream)
                assert torch.equal(got, planes)
        except Exception as e:  # noqa: BLE001
            errors.append((W, repr(e)))

    threads = [threading.Thread(target=work, args=(W,)) for W in (40, 700, 2048, 4000)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
