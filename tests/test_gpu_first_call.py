"""The first call of a length, which makes the length's table, on a stream that
is not ordered behind the legacy default stream: mixed and prime radices,
Bluestein in one kernel and in several, two kernels, and an uneven batch."""
import math

import numpy as np
import pytest

import seeded_inputs as si
from tests.gpu_util import c64_from_dev, c64_to_dev, fft_rel_err

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def bp():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2310_16214_gb300 as bp
    return bp


@pytest.mark.parametrize("n", [11250, 9856, 4007, 4127, 1 << 17])
def test_first_call_on_a_side_stream(bp, n):
    x = si.fft_c64(3, n, stream=2700 + n)
    xd = c64_to_dev(x)
    out = torch.empty_like(xd)
    torch.cuda.synchronize()
    side = torch.cuda.Stream()
    with torch.cuda.stream(side):
        bp.fft_batched(xd, out, n, 3, -1)
    side.synchronize()
    ref = np.fft.fft(x.astype(np.complex128), axis=1)
    assert fft_rel_err(c64_from_dev(out).reshape(3, n), ref).max() <= 1e-5 * math.ceil(math.log2(n))


def test_uneven_batch_on_a_side_stream(bp):
    z = [si.fft_c64(1, 1 << e, stream=2800 + e) for e in range(5, 14)]
    ins = [c64_to_dev(v) for v in z]
    outs = [torch.empty_like(v) for v in ins]
    torch.cuda.synchronize()
    side = torch.cuda.Stream()
    with torch.cuda.stream(side):
        batch = bp.UnevenBatch([{"op": bp.OP_FFT, "n": v.shape[1], "in": [i], "out": o, "dir": -1}
                                for v, i, o in zip(z, ins, outs)])
        batch.launch()
    side.synchronize()
    for v, o in zip(z, outs):
        ref = np.fft.fft(v.astype(np.complex128), axis=1)
        assert fft_rel_err(c64_from_dev(o), ref).max() <= 1e-5 * math.log2(v.shape[1])
