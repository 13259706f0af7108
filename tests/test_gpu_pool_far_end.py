"""Max-pooling of outputs with 2^31 and more 16-byte vectors: the result, and that it stays on 16-byte vectors."""
import pytest
import torch

from paper_1908_11263_gb300 import qnn

pytestmark = pytest.mark.gpu


def _ms(x, out):
    start, end = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    start.record()
    qnn.maxpool(x, 1, 1, 8, out=out)
    end.record()
    end.synchronize()
    return start.elapsed_time(end)


def test_vectors_past_two_to_the_31():
    qnn.load(build_if_missing=True)
    torch.cuda.set_device(0)
    n, side, c = 2049, 1024, 16
    if torch.cuda.mem_get_info()[0] < 80 << 30:
        pytest.skip("needs 80 GB of free device memory")
    g = torch.Generator(device="cuda").manual_seed(5)
    x = torch.empty((n, side, side, c), device="cuda", dtype=torch.uint8)
    for i in range(0, n, 64):
        part = x[i:i + 64]
        part.copy_(torch.randint(0, 256, part.shape, device="cuda", dtype=torch.uint8, generator=g))
    out = torch.zeros_like(x)
    assert n * side * side * c // 16 >= 1 << 31
    _ms(x, out)
    for i in range(0, n, 64):
        assert torch.equal(out[i:i + 64], x[i:i + 64])
    # 2047 images stay below 2^31 vectors; byte by byte the larger tensor took 20 times as long
    below = min(_ms(x[:2047], out[:2047]) for _ in range(3))
    assert min(_ms(x, out) for _ in range(3)) < 3 * below
    del x, out
    torch.cuda.empty_cache()
