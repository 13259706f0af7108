"""Chains of overlapped launches on one stream: each reads what the launches before it wrote."""
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


def test_workspace_copied_two_launches_before_the_run():
    """A prepared image moved by one of the library's own (overlapping) kernels, another short launch, then the
    run that reads the image ahead of its wait: the layers alternate, so a stale image shows."""
    rng = np.random.default_rng(11)
    n, h, w, c, m = 2, 16, 16, 32, 64
    x = rng.integers(0, 256, size=(n, h, w, c))
    layers = []
    for _ in range(2):
        wt = rng.integers(-128, 128, size=(m, 3, 3, c))
        kappa = rng.integers(1, 65, size=m).astype(np.int16)
        lam = rng.integers(-(1 << 15), 1 << 15, size=m).astype(np.int32)
        conv = qnn.PreparedConv(to_dev(wt, torch.int8), to_dev(kappa, torch.int16), to_dev(lam, torch.int32), n=n,
                                h=h, wd=w, shift=12, pad=1)
        assert qnn.tc_kernel(conv.desc) == qnn.ALGO_TC_WINDOW
        layers.append((conv, conv_oracle(x, wt, None, kappa, lam, None, 12, 8, (1, 1), (1, 1))))
    xd = to_dev(x, torch.uint8)
    images = [conv.workspace.clone() for conv, _ in layers]
    run = layers[0][0]
    # (a long launch ahead, so that the copy still waits for it when the launches after it are queued)
    big = torch.zeros(256 << 20, dtype=torch.int8, device="cuda")
    small = torch.zeros(4096, dtype=torch.int8, device="cuda")
    packed, packed_small = qnn.pack_subbyte(big, 2), qnn.pack_subbyte(small, 2)
    for i in range(32):
        qnn.pack_subbyte(big, 2, out=packed)
        qnn.pack_subbyte(images[i % 2].view(torch.int8), 8, out=run.workspace)
        qnn.pack_subbyte(small, 2, out=packed_small)
        got = run(xd).cpu().numpy().reshape(-1)
        assert first_mismatch(got, layers[i % 2][1]) is None
    qnn.device_status()
