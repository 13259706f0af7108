"""GPU parity of packing, unpacking and max-pooling at the edges of their vector groups, byte for byte
against the oracle."""
import numpy as np
import pytest
import torch

import oracle
from paper_1908_11263_gb300 import qnn

from gpu_util import check_guard, dev, guarded_output, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def loaded():
    qnn.load(build_if_missing=True)
    torch.cuda.set_device(0)


@pytest.mark.parametrize("bits", [8, 4, 2])
@pytest.mark.parametrize("count", [8, 16, 24, 16 * 1024, 16 * 1024 + 8, 16 * 4096 * 3 + 40])
@pytest.mark.parametrize("offset", [0, 4])
def test_pack_unpack_edges(bits, count, offset):
    """Whole groups of 16 values, a rest, and tensors that start off a group's alignment."""
    rng = np.random.default_rng(count + bits + offset)
    v = rng.integers(-128, 128, size=count).astype(np.int8)  # only the low Q bits count
    src = torch.empty(count + offset, dtype=torch.int8, device=dev())
    src[offset:] = to_dev(v)
    packed, buf = guarded_output((count * bits // 8,))
    qnn.pack_subbyte(src[offset:], bits, out=packed)
    check_guard(buf)
    want = oracle.pack((v.astype(np.int64) & ((1 << bits) - 1)), bits) if bits < 8 else v.view(np.uint8)
    np.testing.assert_array_equal(packed.cpu().numpy(), want)
    psrc = torch.empty(want.size + offset, dtype=torch.uint8, device=dev())
    psrc[offset:] = packed
    for signed in (False, True):
        whole = torch.full((count + offset + 64,), 0x5A, dtype=torch.int8, device=dev())
        qnn.unpack_subbyte(psrc[offset:], bits, signed, out=whole[offset:offset + count])
        got = whole.cpu().numpy()
        assert np.all(got[:offset] == 0x5A) and np.all(got[offset + count:] == 0x5A)
        if bits < 8:
            np.testing.assert_array_equal(got[offset:offset + count].astype(np.int64), oracle.unpack(want, count, bits, signed))
        else:
            np.testing.assert_array_equal(got[offset:offset + count], v)


@pytest.mark.parametrize("bits,n,h,w,c,k,s", [(8, 1, 2, 2, 16, 2, 2), (8, 5, 31, 17, 48, 2, 2), (4, 3, 9, 11, 96, 2, 1),
                                              (2, 7, 13, 6, 128, 3, 2), (2, 2, 5, 5, 64, 5, 1), (8, 2, 6, 7, 32, 1, 3)])
def test_maxpool_vectors(bits, n, h, w, c, k, s):
    rng = np.random.default_rng(n + h + c)
    x = rng.integers(0, 1 << bits, size=(n, h, w, c))
    xp = oracle.pack(x.reshape(-1), bits) if bits < 8 else x.astype(np.uint8).reshape(-1)
    want = oracle.maxpool(xp, n, h, w, c, k, s, bits)
    out, buf = guarded_output((n, (h - k) // s + 1, (w - k) // s + 1, c * bits // 8))
    qnn.maxpool(torch.from_numpy(xp).to(dev()).view(n, h, w, c * bits // 8), k, s, bits, out=out)
    check_guard(buf)
    np.testing.assert_array_equal(out.cpu().numpy().reshape(-1), want)
