"""GPU parity of the gather kernel (the default of INT-8 layers that the window kernel does not take:
strides, odd channel counts and widths, wide layers), byte for byte against the oracle."""
import numpy as np
import pytest
import torch

from paper_1908_11263_gb300 import qnn

from gpu_util import check_guard, conv_gpu, conv_oracle, first_mismatch, guarded_output, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def loaded():
    qnn.load(build_if_missing=True)
    torch.cuda.set_device(0)


def _case(seed, n, h, w, c, m, kh, kw):
    """Random layer whose outputs spread over the byte range; one channel's constants need 64 bits."""
    rng = np.random.default_rng(seed)
    x = rng.integers(0, 256, size=(n, h, w, c))
    wt = rng.integers(-128, 128, size=(m, kh, kw, c))
    bias = rng.integers(-4096, 4097, size=m).astype(np.int32)
    kappa = rng.integers(-64, 65, size=m).astype(np.int16)
    lam = rng.integers(-(1 << 15), (1 << 15) + 1, size=m).astype(np.int32)
    shift = int(np.ceil(np.log2(max(1.0, 2 * np.sqrt(kh * kw * c) * 147 * 74 * 33 / 255))))
    shifts = (shift + rng.integers(-1, 2, size=m)).astype(np.uint8)
    kappa[0], lam[0] = 32767, (1 << 31) - 1
    return x, wt, bias, kappa, lam, shifts, shift


# (n, h, w, c, m, kh, kw, stride, pad): one and several tiles of 128 pixels with ragged ends, filters kept, converted
# per slab (m over 128, long kernels) and in one or several exact chunks, aligned and byte-wise granules
PACKED = [
    (2, 16, 16, 32, 64, 3, 3, (2, 2), (1, 1)),
    (1, 17, 15, 16, 32, 3, 3, (2, 1), (1, 1)),
    (3, 33, 45, 20, 44, 3, 3, (1, 1), (1, 1)),
    (2, 19, 21, 3, 10, 5, 5, (2, 2), (2, 2)),
    (1, 1, 1, 1, 1, 1, 1, (1, 1), (0, 0)),
    (1, 7, 9, 17, 33, 3, 2, (3, 2), (2, 4)),
    (2, 30, 28, 64, 128, 3, 3, (2, 2), (1, 1)),
    (1, 13, 11, 256, 160, 3, 3, (2, 2), (1, 1)),
    (1, 9, 13, 45, 130, 5, 3, (1, 1), (2, 1)),
    (1, 11, 11, 80, 96, 3, 3, (2, 2), (0, 0)),
    (2, 9, 9, 128, 64, 3, 3, (2, 2), (1, 1)),
    (1, 12, 13, 129, 31, 3, 3, (1, 1), (1, 1)),
    (1, 5, 3, 7, 300, 1, 1, (1, 1), (3, 0)),
]


@pytest.mark.parametrize("shape", PACKED, ids=lambda s: "x".join(str(v) for v in s[:7]) + f"_s{s[7][0]}{s[7][1]}")
def test_packed_filters(shape):
    n, h, w, c, m, kh, kw, stride, pad = shape
    x, wt, bias, kappa, lam, shifts, shift = _case(sum(shape[:7]), n, h, w, c, m, kh, kw)
    want = conv_oracle(x, wt, bias, kappa, lam, shifts, shift, 8, stride, pad)
    got = conv_gpu(x, wt, bias, kappa, lam, shifts, shift, 8, stride, pad, qnn.ALGO_AUTO)
    assert first_mismatch(got, want) is None, first_mismatch(got, want)
    want = conv_oracle(x, wt, None, kappa, lam, None, shift, 8, stride, pad)
    got = conv_gpu(x, wt, None, kappa, lam, None, shift, 8, stride, pad, qnn.ALGO_AUTO)
    assert first_mismatch(got, want) is None, first_mismatch(got, want)


# (n, h, w, c, m, k, pad): stride-1 layers past the window kernel's limits
WIDE = [
    (1, 6, 6, 256, 256, 3, 1),
    (3, 14, 14, 128, 136, 3, 1),
    (2, 14, 14, 256, 512, 1, 0),
    (5, 7, 8, 80, 32, 3, 1),
    (1, 16, 5, 96, 48, 5, 2),
    (1, 1, 1, 64, 160, 1, 0),
    (2, 10, 13, 112, 257, 1, 0),
]


@pytest.mark.parametrize("shape", WIDE, ids=lambda s: "x".join(str(v) for v in s))
def test_prepared_and_one_shot_wide_layers(shape):
    n, h, w, c, m, k, pad = shape
    x, wt, bias, kappa, lam, shifts, shift = _case(sum(shape), n, h, w, c, m, k, k)
    want = conv_oracle(x, wt, bias, kappa, lam, shifts, shift, 8, (1, 1), (pad, pad))
    got = conv_gpu(x, wt, bias, kappa, lam, shifts, shift, 8, (1, 1), (pad, pad), qnn.ALGO_AUTO)
    assert first_mismatch(got, want) is None, first_mismatch(got, want)
    conv = qnn.PreparedConv(to_dev(wt, torch.int8), to_dev(kappa, torch.int16), to_dev(lam, torch.int32), n=n, h=h,
                            wd=w, bias=to_dev(bias, torch.int32), shifts=to_dev(shifts, torch.uint8), shift=shift,
                            pad=pad)
    out, buf = guarded_output(conv.out_shape)
    for _ in range(2):
        conv(to_dev(x, torch.uint8), out=out)
    qnn.device_status()
    check_guard(buf)
    got = out.cpu().numpy().reshape(-1)
    assert first_mismatch(got, want) is None, first_mismatch(got, want)


@pytest.mark.parametrize("xval,wval", [(0, -128), (255, 127), (255, -128), (0, 127)])
@pytest.mark.parametrize("c,stride", [(64, 2), (128, 2), (256, 2), (256, 1)])
def test_exact_at_the_bounds(xval, wval, c, stride):
    """Constant layers drive every accumulator chunk to its extreme (1024 products of 2^14); with kappa = 1,
    shift = 0 and lambda = 100 - acc each output reads 100 only if acc is exact."""
    x = np.full((1, 9, 9, c), xval)
    wt = np.full((130, 3, 3, c), wval)
    wt[1::2] = np.clip(-wt[1::2], -128, 127)
    acc = (xval * wt.reshape(130, -1).sum(axis=1)).astype(np.int64)
    got = conv_gpu(x, wt, None, np.ones(130, np.int16), (100 - acc).astype(np.int32), None, 0, 8, (stride, stride),
                   (0, 0), qnn.ALGO_AUTO)
    assert np.all(got == 100), np.unique(got)
