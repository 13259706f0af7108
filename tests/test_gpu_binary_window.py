"""GPU parity of the INT-1 layers that the window kernel takes, byte for byte against the oracle."""
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


def _bits(v):
    return np.packbits(np.asarray(v, np.uint8).reshape(-1), bitorder="little")


# (n, h, w, c, m, kh, kw, pad): one and two strips, several tiles across (whole rows are read for each), partial tiles,
# 32 to 128 filters, all channel counts of the kernel, rectangular kernels
BINARY = [
    (2, 16, 16, 32, 64, 3, 3, 1),
    (1, 7, 40, 32, 8, 3, 3, 1),
    (3, 33, 28, 64, 72, 5, 5, 2),
    (1, 18, 12, 96, 128, 3, 3, 0),
    (2, 5, 4, 128, 24, 1, 1, 0),
    (1, 20, 24, 128, 104, 3, 3, 1),
    (1, 17, 20, 32, 32, 8, 8, 4),
    (300, 9, 8, 32, 40, 2, 4, 1),
]


@pytest.mark.parametrize("shape", BINARY, ids=lambda s: "x".join(str(v) for v in s))
@pytest.mark.parametrize("extreme", [False, True])
def test_binary(shape, extreme):
    n, h, w, c, m, kh, kw, pad = shape
    rng = np.random.default_rng(sum(shape))
    xb, wb = rng.integers(0, 2, size=(n, h, w, c)), rng.integers(0, 2, size=(m, kh, kw, c))
    kk = kh * kw * c
    tau = rng.integers(kk // 2 - int(np.sqrt(kk)), kk // 2 + int(np.sqrt(kk)) + 1, size=m).astype(np.int32)
    if extreme:  # always and never reached, and the ends of the count
        tau[:8] = [np.iinfo(np.int32).min, np.iinfo(np.int32).max, 0, 1, kk, kk + 1, -1, 1 << 30]
    oh, ow = h + 2 * pad - kh + 1, w + 2 * pad - kw + 1
    shp = dict(n=n, h=h, w=w, c=c, m=m, kh=kh, kw=kw, sh=1, sw=1, ph=pad, pw=pad)
    want = oracle.conv_binary(_bits(xb), _bits(wb), shp, tau)
    xd = torch.from_numpy(_bits(xb)).to(dev()).view(n, h, w, c // 8)
    wd = torch.from_numpy(_bits(wb)).to(dev()).view(m, kh, kw, c // 8)
    out, buf = guarded_output((n, oh, ow, m // 8))
    qnn.conv_binary(xd, wd, torch.from_numpy(tau).to(dev()), pad=pad, out=out)
    qnn.device_status()
    check_guard(buf)
    assert first_mismatch(out.cpu().numpy().reshape(-1), want) is None
