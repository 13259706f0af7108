"""GPU parity of layers at the lines between kernels, byte for byte against the oracle, each with the kernel it has to
run on."""
import numpy as np
import pytest
import torch

import oracle
from paper_1908_11263_gb300 import qnn

from gpu_util import check_guard, dev, first_mismatch, guarded_output

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def loaded():
    qnn.load(build_if_missing=True)
    torch.cuda.set_device(0)


def _name(s):
    return "x".join(str(v) for v in s)


def _bits(v):
    return np.packbits(np.asarray(v, np.uint8).reshape(-1), bitorder="little")


WINDOW, COUNT, STACKED = qnn.KERNEL_WINDOW, qnn.KERNEL_COUNT, qnn.KERNEL_WINDOW | qnn.KERNEL_STACKED
# (n, h, w, c, m, kh, kw, pad): few products per output on the window kernel, few filters, one and two strips, several
# tiles across, stacked images; the same just below the line on the counts
BINARY = [
    ((1, 7, 40, 32, 24, 3, 3, 1), WINDOW),
    ((2, 5, 4, 128, 48, 1, 1, 0), WINDOW),
    ((2, 5, 4, 128, 40, 1, 1, 0), COUNT),
    ((3, 20, 24, 64, 96, 1, 1, 0), WINDOW),
    ((1, 9, 16, 96, 64, 1, 1, 0), WINDOW),
    ((2, 33, 28, 32, 8, 5, 5, 2), WINDOW),
    ((2, 33, 28, 32, 8, 4, 5, 2), COUNT),
    ((170, 20, 40, 64, 16, 3, 3, 0), STACKED),
    ((400, 9, 24, 96, 72, 1, 1, 0), STACKED),
]


@pytest.mark.parametrize("shape,kernel", BINARY, ids=lambda v: _name(v) if isinstance(v, tuple) else str(v))
def test_binary(shape, kernel):
    n, h, w, c, m, kh, kw, pad = shape
    assert qnn.kernel(qnn.conv_desc(n, h, w, c, m, kh, kw, 1, pad, 1))[0] == kernel
    rng = np.random.default_rng(sum(shape))
    xb, wb = rng.integers(0, 2, size=(n, h, w, c)), rng.integers(0, 2, size=(m, kh, kw, c))
    kk = kh * kw * c
    tau = rng.integers(kk // 2 - int(np.sqrt(kk)), kk // 2 + int(np.sqrt(kk)) + 1, size=m).astype(np.int32)
    oh, ow = h + 2 * pad - kh + 1, w + 2 * pad - kw + 1
    want = oracle.conv_binary(_bits(xb), _bits(wb), dict(n=n, h=h, w=w, c=c, m=m, kh=kh, kw=kw, sh=1, sw=1, ph=pad, pw=pad),
                              tau)
    out, buf = guarded_output((n, oh, ow, m // 8))
    qnn.conv_binary(torch.from_numpy(_bits(xb)).to(dev()).view(n, h, w, c // 8),
                    torch.from_numpy(_bits(wb)).to(dev()).view(m, kh, kw, c // 8), torch.from_numpy(tau).to(dev()), pad=pad,
                    out=out)
    qnn.device_status()
    check_guard(buf)
    assert first_mismatch(out.cpu().numpy().reshape(-1), want) is None


# (n, h, w, c, m, k, pad, bits, stacked): a round saved of a few (short INT-8 filters keep the plain form), of many
@pytest.mark.parametrize("n,h,w,c,m,k,pad,bits,stacked", [
    (2048, 14, 14, 32, 64, 3, 1, 8, False), (1003, 57, 8, 16, 32, 3, 1, 8, False), (691, 45, 8, 32, 16, 1, 0, 8, False),
    (2048, 14, 14, 32, 64, 3, 1, 4, True), (256, 56, 56, 64, 64, 3, 1, 8, True), (1024, 8, 8, 32, 64, 5, 2, 8, True),
    (331, 7, 12, 32, 24, 3, 1, 8, True), (366, 44, 8, 16, 104, 3, 1, 8, True), (512, 16, 16, 32, 64, 3, 1, 8, False)])
def test_stacked_line(n, h, w, c, m, k, pad, bits, stacked):
    if torch.cuda.get_device_properties(0).multi_processor_count != 152:
        pytest.skip("rounds of 152 blocks")
    d = qnn.conv_desc(n, h, w, c, m, k, k, 1, pad, bits)
    for prepared in (False, True):
        assert qnn.kernel(d, prepared)[0] == (STACKED if stacked else WINDOW)
