"""The window kernel on stacked images (tiles that run across the images of a batch), byte for byte against the oracle,
in every form that takes them: one-shot, prepared, with the fused pool, with thresholds, INT-1."""
import numpy as np
import pytest
import torch

import oracle
from paper_1908_11263_gb300 import qnn

from gpu_util import (check_guard, conv_gpu, conv_oracle, dev, first_mismatch, guarded_output, pack_gpu, to_dev)

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def loaded():
    qnn.load(build_if_missing=True)
    torch.cuda.set_device(0)


# (n, h, w, c, m, k, pad, bits): more than one tile per SM, so that stacked images are chosen; a tile over two to nine
# images, an odd number of rows per image (even with the pool), the last image alone in its tile, rows that end at a
# tile's edge, several tiles across (row segments; whole rows), no padding, folded kernel columns, one and two strips
LAYERS = [
    (400, 8, 8, 16, 16, 5, 2, 8),
    (331, 7, 12, 32, 24, 3, 1, 8),
    (163, 17, 16, 16, 40, 3, 1, 8),
    (700, 2, 16, 16, 8, 1, 0, 8),
    (611, 1, 16, 32, 8, 3, 1, 8),
    (90, 18, 40, 16, 8, 3, 1, 8),
    (170, 20, 16, 24, 16, 5, 0, 8),
    (120, 21, 32, 3, 16, 5, 2, 8),
    (347, 9, 12, 32, 64, 3, 1, 4),
    (331, 14, 16, 64, 8, 3, 1, 2),
    (160, 19, 32, 32, 16, 3, 1, 2),
]


@pytest.mark.parametrize("layer", LAYERS, ids=lambda s: "x".join(str(v) for v in s))
def test_stacked(layer):
    n, h, w, c, m, k, pad, bits = layer
    rng = np.random.default_rng(sum(layer))
    top, half, per = (1 << bits) - 1, 1 << (bits - 1), 8 // bits
    x = rng.integers(0, top + 1, size=(n, h, w, c))
    wt = rng.integers(-half, half, size=(m, k, k, c))
    acc = oracle.conv_acc(x[:8], wt, (1, 1), (pad, pad)).reshape(-1, m)
    bias = (-acc.mean(axis=0)).astype(np.int32)
    kappa = rng.integers(-64, 65, size=m).astype(np.int16)
    lam = rng.integers(-16, 17, size=m).astype(np.int32)
    shift = max(0, int(np.ceil(np.log2(1.6 * acc.std() * 32 / top))))
    want = conv_oracle(x, wt, bias, kappa, lam, None, shift, bits, (1, 1), (pad, pad))
    got = conv_gpu(x, wt, bias, kappa, lam, None, shift, bits, (1, 1), (pad, pad), qnn.ALGO_AUTO)
    assert first_mismatch(got, want) is None, first_mismatch(got, want)
    xd = pack_gpu(x, bits).view(n, h, w, c // per)
    wd = pack_gpu(wt, bits).view(m, k, k, c // per)
    wd = wd.view(torch.int8) if bits == 8 else wd
    desc = qnn.conv_desc(n, h, w, c, m, k, k, 1, pad, bits, shift)
    oh, ow = h + 2 * pad - k + 1, w + 2 * pad - k + 1
    if qnn.tc_kernel(desc) == qnn.ALGO_TC_WINDOW:
        conv = qnn.PreparedConv(wd, to_dev(kappa, torch.int16), to_dev(lam, torch.int32), n=n, h=h, wd=w,
                                bias=to_dev(bias, torch.int32), shift=shift, bits=bits, pad=pad)
        out, buf = guarded_output(conv.out_shape)
        conv(xd, out=out)
        qnn.device_status()
        check_guard(buf)
        assert first_mismatch(out.cpu().numpy().reshape(-1), want) is None
        if oh > 1 and ow > 1:
            out, buf = guarded_output((n, oh // 2, ow // 2, m // per))
            conv.pool2(xd, out=out)
            qnn.device_status()
            check_guard(buf)
            assert first_mismatch(out.cpu().numpy().reshape(-1), oracle.maxpool(want, n, oh, ow, m, 2, 2, bits)) is None
    if bits < 8:
        thr = np.stack([np.quantile(acc, (q + 0.5) / top, axis=0) for q in range(top)], axis=1).astype(np.int32)
        out = qnn.conv_hwc_thresholds(xd, wd, to_dev(thr, torch.int32), bits=bits, pad=pad)
        qnn.device_status()
        acc = oracle.conv_acc(x, wt, (1, 1), (pad, pad)).reshape(-1, m)
        want = oracle.pack((thr[None, :, :] <= acc[:, :, None]).sum(axis=2).reshape(-1), bits)
        assert first_mismatch(out.cpu().numpy().reshape(-1), want) is None


@pytest.mark.parametrize("shape", [(331, 7, 12, 32, 40, 3, 1), (170, 18, 40, 64, 8, 3, 0), (420, 6, 4, 128, 72, 5, 2)],
                         ids=lambda s: "x".join(str(v) for v in s))
def test_stacked_binary(shape):
    n, h, w, c, m, k, pad = shape
    rng = np.random.default_rng(sum(shape))
    xb, wb = rng.integers(0, 2, size=(n, h, w, c)), rng.integers(0, 2, size=(m, k, k, c))
    kk = k * k * c
    tau = rng.integers(kk // 2 - int(np.sqrt(kk)), kk // 2 + int(np.sqrt(kk)) + 1, size=m).astype(np.int32)
    oh, ow = h + 2 * pad - k + 1, w + 2 * pad - k + 1
    x, wt = (np.packbits(v.astype(np.uint8).reshape(-1), bitorder="little") for v in (xb, wb))
    want = oracle.conv_binary(x, wt, dict(n=n, h=h, w=w, c=c, m=m, kh=k, kw=k, sh=1, sw=1, ph=pad, pw=pad), tau)
    out, buf = guarded_output((n, oh, ow, m // 8))
    qnn.conv_binary(torch.from_numpy(x).to(dev()).view(n, h, w, c // 8), torch.from_numpy(wt).to(dev()).view(m, k, k, c // 8),
                    torch.from_numpy(tau).to(dev()), pad=pad, out=out)
    qnn.device_status()
    check_guard(buf)
    assert first_mismatch(out.cpu().numpy().reshape(-1), want) is None
