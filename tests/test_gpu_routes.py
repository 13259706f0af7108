"""GPU parity of layers at the lines between kernels, byte for byte against the oracle, each with the kernel it has to
run on."""
import numpy as np
import pytest
import torch

import oracle
from paper_1908_11263_gb300 import qnn

from gpu_util import check_guard, conv_gpu, conv_oracle, dev, first_mismatch, guarded_output, to_dev

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
    ((150, 36, 20, 96, 8, 3, 3, 1), COUNT),
    ((9, 16, 36, 64, 16, 3, 3, 1), WINDOW),
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


def _layer(seed, n, h, w, c, m, kh, kw):
    """Random INT-8 layer whose outputs spread over the byte range; one channel's constants need 64 bits."""
    rng = np.random.default_rng(seed)
    x, wt = rng.integers(0, 256, size=(n, h, w, c)), rng.integers(-128, 128, size=(m, kh, kw, c))
    bias = rng.integers(-4096, 4097, size=m).astype(np.int32)
    kappa = rng.integers(-64, 65, size=m).astype(np.int16)
    lam = rng.integers(-(1 << 15), (1 << 15) + 1, size=m).astype(np.int32)
    shift = int(np.ceil(np.log2(max(1.0, 2 * np.sqrt(kh * kw * c) * 147 * 74 * 33 / 255))))
    shifts = (shift + rng.integers(-1, 2, size=m)).astype(np.uint8)
    kappa[0], lam[0] = 32767, (1 << 31) - 1
    return x, wt, bias, kappa, lam, shifts


DIRECT, GATHER = qnn.KERNEL_DIRECT, qnn.KERNEL_GATHER
# (n, h, w, c, m, kh, kw, stride, pad): the smallest layer and three channel blocks on packed filters; few loads per
# output and many outputs, words and bytes, on either side of the line to the CUDA cores
SMALL = [
    ((1, 1, 1, 21, 1, 1, 1, 1, 0), GATHER),
    ((1, 5, 3, 21, 300, 1, 1, 1, 3), GATHER),
    ((1, 7, 9, 3, 5, 3, 3, 2, 1), GATHER),
    ((12, 41, 5, 4, 13, 3, 4, 2, 1), GATHER),
    ((12, 40, 44, 16, 100, 2, 2, 2, 0), GATHER),
    ((1, 1, 1, 1, 1, 1, 1, 1, 0), DIRECT),
    ((50, 60, 29, 3, 23, 1, 1, 1, 0), DIRECT),
    ((36, 10, 58, 1, 11, 3, 3, 1, 1), DIRECT),
    ((8, 42, 16, 16, 5, 1, 1, 3, 0), DIRECT),
    ((5, 9, 11, 8, 2, 2, 2, 2, 1), DIRECT),
]


@pytest.mark.parametrize("shape,kernel", SMALL, ids=lambda v: _name(v) if isinstance(v, tuple) else str(v))
def test_small_layers(shape, kernel):
    n, h, w, c, m, kh, kw, stride, pad = shape
    assert qnn.kernel(qnn.conv_desc(n, h, w, c, m, kh, kw, stride, pad))[0] == kernel
    x, wt, bias, kappa, lam, shifts = _layer(sum(shape), n, h, w, c, m, kh, kw)
    want = conv_oracle(x, wt, bias, kappa, lam, shifts, 0, 8, (stride, stride), (pad, pad))
    got = conv_gpu(x, wt, bias, kappa, lam, shifts, 0, 8, (stride, stride), (pad, pad), qnn.ALGO_AUTO)
    assert first_mismatch(got, want) is None, first_mismatch(got, want)


@pytest.mark.parametrize("per_channel", [True, False])
def test_gather_long_shifts(per_channel):
    """Shifts from 0 to 62 in the gather kernel's 32-bit form (kappa small enough for it)."""
    n, h, w, c, m = 2, 9, 9, 24, 64
    assert qnn.kernel(qnn.conv_desc(n, h, w, c, m, 3, 3, 2, 1))[0] == GATHER
    x, wt, bias, _, lam, _ = _layer(7, n, h, w, c, m, 3, 3)
    kappa = np.where(np.arange(m) % 2, 1, -1).astype(np.int16)
    lam = np.where(np.arange(m) % 3, 100, -100).astype(np.int32)
    for shift in (0, 31, 32, 40, 62):
        shifts = ((np.arange(m) + shift) % 63).astype(np.uint8) if per_channel else None
        want = conv_oracle(x, wt, bias, kappa, lam, shifts, shift, 8, (2, 2), (1, 1))
        got = conv_gpu(x, wt, bias, kappa, lam, shifts, shift, 8, (2, 2), (1, 1), qnn.ALGO_AUTO)
        assert first_mismatch(got, want) is None, (shift, first_mismatch(got, want))


GENERAL = qnn.KERNEL_GENERAL
# (n, h, w, c, m, k, pad), prepared kernel, one-shot kernel: long kernels (more than 16 taps) of 64-channel steps, few
# filters kept in shared memory, a preparation that only the general kernel starts beside, and the gather kernel's
WIDE = [
    ((2, 6, 6, 256, 16, 5, 2), GENERAL, GENERAL),
    ((3, 7, 7, 192, 40, 7, 3), GENERAL, GENERAL),
    ((2, 9, 8, 320, 88, 5, 2), GENERAL, GENERAL),
    ((4, 8, 8, 80, 8, 3, 1), GATHER, GENERAL),
    ((5, 7, 7, 256, 16, 3, 1), GENERAL, GENERAL),
    ((2, 9, 8, 160, 88, 5, 2), GATHER, GATHER),
    ((3, 14, 14, 128, 136, 3, 1), GATHER, GATHER),
    ((2, 7, 6, 64, 192, 1, 0), GATHER, GATHER),
]


@pytest.mark.parametrize("shape,prepared,one_shot", WIDE, ids=lambda v: _name(v) if isinstance(v, tuple) else str(v))
def test_wide_layers(shape, prepared, one_shot):
    n, h, w, c, m, k, pad = shape
    d = qnn.conv_desc(n, h, w, c, m, k, k, 1, pad)
    assert (qnn.kernel(d, True)[0], qnn.kernel(d)[0]) == (prepared, one_shot)
    x, wt, bias, kappa, lam, shifts = _layer(sum(shape), n, h, w, c, m, k, k)
    want = conv_oracle(x, wt, bias, kappa, lam, shifts, 0, 8, (1, 1), (pad, pad))
    got = conv_gpu(x, wt, bias, kappa, lam, shifts, 0, 8, (1, 1), (pad, pad), qnn.ALGO_AUTO)
    assert first_mismatch(got, want) is None, first_mismatch(got, want)
    conv = qnn.PreparedConv(to_dev(wt, torch.int8), to_dev(kappa, torch.int16), to_dev(lam, torch.int32), n=n, h=h, wd=w,
                            bias=to_dev(bias, torch.int32), shifts=to_dev(shifts, torch.uint8), pad=pad)
    out, buf = guarded_output(conv.out_shape)
    conv(to_dev(x, torch.uint8), out=out)
    qnn.device_status()
    check_guard(buf)
    assert first_mismatch(out.cpu().numpy().reshape(-1), want) is None


ROWS = qnn.KERNEL_WINDOW | qnn.KERNEL_ROWS
# (n, h, w, c, m, k, bits): images that fill the tiles, badly, badly with few rounds, and badly with byte stores
@pytest.mark.parametrize("n,h,w,c,m,k,bits,want", [
    (734, 13, 48, 32, 120, 3, 2, ROWS), (941, 38, 20, 32, 48, 3, 2, GENERAL), (2, 29, 24, 32, 64, 3, 2, ROWS),
    (529, 11, 36, 32, 120, 3, 2, ROWS), (53, 51, 20, 32, 40, 1, 2, GENERAL), (2, 34, 28, 24, 112, 3, 8, GENERAL),
    (5, 26, 44, 40, 16, 1, 8, ROWS)])
def test_whole_rows_line(n, h, w, c, m, k, bits, want):
    if torch.cuda.get_device_properties(0).multi_processor_count != 152:
        pytest.skip("rounds of 152 blocks")
    d = qnn.conv_desc(n, h, w, c, m, k, k, 1, k // 2, bits)
    assert qnn.kernel(d)[0] & ~qnn.KERNEL_STACKED == want
    assert qnn.kernel(d, prepared=True)[0] == GENERAL


@pytest.mark.parametrize("n,h,w,m,want", [(120, 20, 20, 48, GENERAL), (90, 20, 36, 120, ROWS)])
def test_whole_rows_parity(n, h, w, m, want):
    """INT-2, 3 x 3, on either side of that line."""
    assert qnn.kernel(qnn.conv_desc(n, h, w, 32, m, 3, 3, 1, 1, 2))[0] & ~qnn.KERNEL_STACKED == want
    rng = np.random.default_rng(n + m)
    x, wt = rng.integers(0, 4, size=(n, h, w, 32)), rng.integers(-2, 2, size=(m, 3, 3, 32))
    kappa = rng.integers(-64, 65, size=m).astype(np.int16)
    lam, bias = rng.integers(-500, 500, size=m).astype(np.int32), rng.integers(-30, 30, size=m).astype(np.int32)
    want = conv_oracle(x, wt, bias, kappa, lam, None, 8, 2, (1, 1), (1, 1))
    got = conv_gpu(x, wt, bias, kappa, lam, None, 8, 2, (1, 1), (1, 1), qnn.ALGO_AUTO)
    assert first_mismatch(got, want) is None, first_mismatch(got, want)
