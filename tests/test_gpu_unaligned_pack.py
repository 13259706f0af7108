"""Packing and unpacking at odd addresses around one wave of blocks (where threads start to take a second byte)."""
import pytest
import torch

from paper_1908_11263_gb300 import qnn

from gpu_util import dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def loaded():
    qnn.load(build_if_missing=True)
    torch.cuda.set_device(0)


@pytest.mark.parametrize("bits", [8, 4, 2])
@pytest.mark.parametrize("extra", [-1, 0, 1, 300])
def test_bytes_past_one_wave(bits, extra):
    per = 8 // bits
    nbytes = torch.cuda.get_device_properties(0).multi_processor_count * 2048 + extra
    count = nbytes * per
    g = torch.Generator(device=dev()).manual_seed(bits * 1000 + extra + 1)
    src = torch.randint(-128, 128, (count + 1,), device=dev(), dtype=torch.int8, generator=g)[1:]
    packed = torch.full((nbytes + 2,), 0xA5, device=dev(), dtype=torch.uint8)
    qnn.pack_subbyte(src, bits, out=packed[1:-1])
    fields = (src.view(torch.uint8) & ((1 << bits) - 1)).view(nbytes, per)
    want = torch.zeros(nbytes, device=dev(), dtype=torch.uint8)
    for k in range(per):
        want |= fields[:, k] << (k * bits)
    assert torch.equal(packed[1:-1], want) and packed[0] == 0xA5 and packed[-1] == 0xA5
    for signed in (False, True):
        back = torch.full((count + 2,), 0x5A, device=dev(), dtype=torch.int8)
        qnn.unpack_subbyte(packed[1:-1], bits, signed, out=back[1:-1])
        values = fields.reshape(-1).view(torch.int8)
        if signed:
            values = (values << (8 - bits)) >> (8 - bits)
        assert torch.equal(back[1:-1], values) and back[0] == 0x5A and back[-1] == 0x5A
