"""Prepared filters do not depend on the batch: layers that one batch size runs on the gather kernel and another on the
general kernel share one workspace."""
import ctypes

import numpy as np
import pytest
import torch

from paper_1908_11263_gb300 import qnn

from gpu_util import conv_oracle, first_mismatch, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def loaded():
    qnn.load(build_if_missing=True)
    torch.cuda.set_device(0)


# (h, w, c, m, k, pad)
@pytest.mark.parametrize("layer", [(6, 6, 80, 40, 3, 1), (4, 4, 192, 40, 5, 2), (7, 7, 256, 16, 3, 1), (5, 6, 64, 300, 1, 0)],
                         ids=lambda s: "x".join(str(v) for v in s))
def test_one_workspace_for_both_kernels(layer):
    h, w, c, m, k, pad = layer
    rng = np.random.default_rng(sum(layer))
    wt = rng.integers(-128, 128, size=(m, k, k, c))
    kappa = rng.integers(-64, 65, size=m).astype(np.int16)
    lam = rng.integers(-(1 << 15), 1 << 15, size=m).astype(np.int32)
    bias = rng.integers(-4096, 4097, size=m).astype(np.int32)
    kappa[0], lam[0] = 32767, (1 << 31) - 1  # 64-bit constants
    shift = 14
    x = rng.integers(0, 256, size=(3, h, w, c))
    want = conv_oracle(x, wt, bias, kappa, lam, None, shift, 8, (1, 1), (pad, pad))
    args = [to_dev(wt, torch.int8), to_dev(kappa, torch.int16), to_dev(lam, torch.int32)]
    kw = dict(h=h, wd=w, bias=to_dev(bias, torch.int32), shift=shift, pad=pad)
    small, general = qnn.PreparedConv(*args, n=3, **kw), qnn.PreparedConv(*args, n=3, algo=qnn.ALGO_TC_GENERAL, **kw)
    large = qnn.PreparedConv(*args, n=1 << 19, **kw)
    assert qnn.kernel(general.desc, True)[0] == qnn.KERNEL_GENERAL
    assert small.nbytes == general.nbytes == large.nbytes
    xd, out = to_dev(x, torch.uint8), torch.empty(want.size, dtype=torch.uint8, device="cuda")
    # every workspace on every kernel
    for conv in (small, general, large):
        for desc in (small.desc, general.desc):
            out.zero_()
            st = qnn.load().qconv_hwc_run(ctypes.byref(desc), xd.data_ptr(), out.data_ptr(), conv.workspace.data_ptr(),
                                          conv.nbytes, torch.cuda.current_stream().cuda_stream)
            assert st == qnn.QNN_OK
            qnn.device_status()
            got = out.cpu().numpy()
            assert first_mismatch(got, want) is None, first_mismatch(got, want)
