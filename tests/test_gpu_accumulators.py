"""GPU parity of the window kernel's accumulators without the pre-load (INT-8 filters too large for
one exact chunk around it) and of its staircase compression, byte for byte against the oracle."""
import numpy as np
import pytest
import torch

import oracle
from paper_1908_11263_gb300 import qnn

from gpu_util import check_guard, conv_gpu, conv_oracle, first_mismatch, guarded_output, pack_gpu, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def loaded():
    qnn.load(build_if_missing=True)
    torch.cuda.set_device(0)


# (n, h, w, c, m, k, pad): one and two accumulators per strip, one and two strips, 32 to 128 filters, table and
# unrolled issue, folded kernel columns (c * k <= 16)
LAYERS = [
    (1, 20, 17 * 2, 64, 64, 3, 1),
    (2, 18, 16, 32, 32, 5, 2),
    (2, 8, 8, 32, 64, 5, 2),
    (1, 16, 16, 32, 128, 3, 1),
    (1, 9, 14, 48, 40, 5, 2),
    (1, 12, 8, 32, 24, 7, 3),
    (2, 17, 32, 3, 32, 5, 2),
]


@pytest.mark.parametrize("wmax", [20, 70, 128], ids=lambda v: f"w{v}")
@pytest.mark.parametrize("layer", LAYERS, ids=lambda s: "x".join(str(v) for v in s))
def test_large_filters(layer, wmax):
    """Filters of magnitude up to wmax with both signs: sums of |w| on both sides of the bounds 2^15 and 2^17.
    Per-channel shifts and one channel that needs 64-bit compression; the one-shot and the prepared launch, the
    latter also with the fused pool."""
    n, h, w, c, m, k, pad = layer
    rng = np.random.default_rng(sum(layer) + wmax)
    x = rng.integers(0, 256, size=(n, h, w, c))
    wt = np.clip(rng.integers(-wmax, wmax + 1, size=(m, k, k, c)), -128, 127)
    bias = rng.integers(-4096, 4097, size=m).astype(np.int32)
    kappa = rng.integers(-64, 65, size=m).astype(np.int16)
    lam = rng.integers(-(1 << 15), (1 << 15) + 1, size=m).astype(np.int32)
    shift = int(np.ceil(np.log2(2 * np.sqrt(k * k * c) * 147 * 0.58 * wmax * 33 / 255)))
    shifts = (shift + rng.integers(-1, 2, size=m)).astype(np.uint8)
    for sh in (shifts, None):
        for wide in (False, True):
            if wide:
                kappa[m // 2], lam[m // 2] = 32767, (1 << 31) - 1
            want = conv_oracle(x, wt, bias, kappa, lam, sh, shift, 8, (1, 1), (pad, pad))
            got = conv_gpu(x, wt, bias, kappa, lam, sh, shift, 8, (1, 1), (pad, pad), qnn.ALGO_TC_WINDOW)
            assert first_mismatch(got, want) is None, first_mismatch(got, want)
            conv = qnn.PreparedConv(to_dev(wt, torch.int8), to_dev(kappa, torch.int16), to_dev(lam, torch.int32), n=n,
                                    h=h, wd=w, bias=to_dev(bias, torch.int32),
                                    shifts=None if sh is None else to_dev(sh, torch.uint8), shift=shift, pad=pad,
                                    algo=qnn.ALGO_TC_WINDOW)
            out, buf = guarded_output(conv.out_shape)
            conv(to_dev(x, torch.uint8), out=out)
            qnn.device_status()
            check_guard(buf)
            assert first_mismatch(out.cpu().numpy().reshape(-1), want) is None
            pooled = conv.pool2(to_dev(x, torch.uint8)).cpu().numpy().reshape(-1)
            want2 = oracle.maxpool(want, n, conv.oh, conv.ow, m, 2, 2, 8)
            assert first_mismatch(pooled, want2) is None, first_mismatch(pooled, want2)


@pytest.mark.parametrize("order", ["sorted", "shuffled", "equal", "ends"])
@pytest.mark.parametrize("bits", [4, 2])
@pytest.mark.parametrize("m", [8, 40, 128])
def test_staircase_orders(bits, m, order):
    """Thresholds in any order, all alike, and at the ends of int32."""
    rng = np.random.default_rng(bits + m)
    n, h, w, c, k = 2, 17, 12, 32, 3
    count, top = (1 << bits) - 1, (1 << bits) - 1
    x = rng.integers(0, top + 1, size=(n, h, w, c))
    wt = rng.integers(-(1 << (bits - 1)), 1 << (bits - 1), size=(m, k, k, c))
    acc = oracle.conv_acc(x, wt, (1, 1), (1, 1)).reshape(-1, m)
    thr = np.stack([np.quantile(acc, (q + 0.5) / count, axis=0) for q in range(count)], axis=1).astype(np.int32)
    if order == "shuffled":
        thr = rng.permuted(thr, axis=1)
    elif order == "equal":
        thr[:] = acc[0][:, None].astype(np.int32)
    elif order == "ends":
        thr[:, 0], thr[:, -1] = np.iinfo(np.int32).min, np.iinfo(np.int32).max
        thr[0, :] = np.iinfo(np.int32).max
        thr[-1, :] = np.iinfo(np.int32).min
    per = 8 // bits
    xd = pack_gpu(x, bits).view(n, h, w, c // per)
    wd = pack_gpu(wt, bits).view(m, k, k, c // per)
    out, buf = guarded_output((n, h, w, m // per))
    qnn.conv_hwc_thresholds(xd, wd, to_dev(thr, torch.int32), bits=bits, pad=1, algo=qnn.ALGO_TC_WINDOW, out=out)
    qnn.device_status()
    check_guard(buf)
    want = oracle.pack((thr[None, :, :] <= acc[:, :, None]).sum(axis=2).reshape(-1), bits)
    assert first_mismatch(out.cpu().numpy().reshape(-1), want) is None


# (n, h, w, c, m, k, pad, bits): several tiles across rows whose pixels are no whole 16-byte units
ROWS = [
    (2, 18, 32, 32, 16, 3, 1, 2),
    (1, 33, 40, 32, 104, 1, 0, 2),
    (1, 9, 36, 96, 24, 3, 1, 2),
    (2, 17, 22, 24, 40, 3, 1, 8),
    (1, 20, 66, 8, 128, 5, 2, 8),
    (3, 7, 34, 40, 64, 3, 0, 8),
]


@pytest.mark.parametrize("layer", ROWS, ids=lambda s: "x".join(str(v) for v in s))
def test_windows_of_whole_rows(layer):
    """One-shot calls, plain, with the fused pool and with thresholds, against the oracle."""
    n, h, w, c, m, k, pad, bits = layer
    rng = np.random.default_rng(sum(layer))
    top, half, per = (1 << bits) - 1, 1 << (bits - 1), 8 // bits
    x = rng.integers(0, top + 1, size=(n, h, w, c))
    wt = rng.integers(-half, half, size=(m, k, k, c))
    acc = oracle.conv_acc(x, wt, (1, 1), (pad, pad)).reshape(-1, m)
    bias = (-acc.mean(axis=0)).astype(np.int32)
    kappa = rng.integers(1, 65, size=m).astype(np.int16)
    lam = rng.integers(-16, 17, size=m).astype(np.int32)
    shift = max(0, int(np.ceil(np.log2(1.6 * acc.std() * 32 / top))))
    want = conv_oracle(x, wt, bias, kappa, lam, None, shift, bits, (1, 1), (pad, pad))
    got = conv_gpu(x, wt, bias, kappa, lam, None, shift, bits, (1, 1), (pad, pad), qnn.ALGO_AUTO)
    assert first_mismatch(got, want) is None, first_mismatch(got, want)
    xd = pack_gpu(x, bits).view(n, h, w, c // per)
    wd = pack_gpu(wt, bits).view(m, k, k, c // per)
    oh, ow = h + 2 * pad - k + 1, w + 2 * pad - k + 1
    pooled = qnn.conv_hwc_pool2(xd, wd.view(torch.int8) if bits == 8 else wd, to_dev(kappa, torch.int16),
                                to_dev(lam, torch.int32), bias=to_dev(bias, torch.int32), shift=shift, bits=bits, pad=pad)
    want2 = oracle.maxpool(want, n, oh, ow, m, 2, 2, bits)
    assert first_mismatch(pooled.cpu().numpy().reshape(-1), want2) is None
    if bits < 8:
        thr = np.stack([np.quantile(acc, (q + 0.5) / top, axis=0) for q in range(top)], axis=1).astype(np.int32)
        out = qnn.conv_hwc_thresholds(xd, wd, to_dev(thr, torch.int32), bits=bits, pad=pad)
        want3 = oracle.pack((thr[None, :, :] <= acc[:, :, None]).sum(axis=2).reshape(-1), bits)
        assert first_mismatch(out.cpu().numpy().reshape(-1), want3) is None
    qnn.device_status()
