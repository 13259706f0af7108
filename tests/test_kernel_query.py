"""qconv_hwc_kernel names the kernel that a call launches and its operand width (no GPU needed)."""
import pytest

from paper_1908_11263_gb300 import build as qbuild
from paper_1908_11263_gb300 import qnn


@pytest.fixture(scope="module", autouse=True)
def lib():
    qbuild.build()
    qnn.load()


def desc(n=1, h=16, w=16, c=32, m=64, k=3, stride=1, pad=1, bits=8, algo=qnn.ALGO_AUTO):
    return qnn.conv_desc(n, h, w, c, m, k, k, stride, pad, bits, 0, algo)


@pytest.mark.parametrize("d,want", [
    (desc(), (qnn.KERNEL_WINDOW, 16)),
    (desc(bits=4), (qnn.KERNEL_WINDOW, 8)),
    (desc(algo=qnn.ALGO_TC_GENERAL), (qnn.KERNEL_GENERAL, 16)),
    (desc(algo=qnn.ALGO_DIRECT), (qnn.KERNEL_DIRECT, 0)),
    (desc(stride=2), (qnn.KERNEL_GATHER, 16)),                     # INT-8, strided
    (desc(h=33, w=45, c=20, m=44), (qnn.KERNEL_GATHER, 16)),       # odd sizes
    (desc(c=128, m=128), (qnn.KERNEL_GATHER, 16)),                 # many channels, prepared filters
    (desc(bits=4, stride=2), (qnn.KERNEL_DIRECT, 0)),
    (desc(bits=1), (qnn.KERNEL_WINDOW, 8)),                        # INT-1 as +1 / -1
    (desc(bits=1, stride=2), (qnn.KERNEL_COUNT, 0)),
], ids=str)
def test_one_shot(d, want):
    kernel, bits = qnn.kernel(d)
    assert (kernel & 0xF, bits) == want


def test_whole_rows_run_on_the_window_kernel_one_shot_only():
    # INT-2 pixels of 8 bytes, image wider than a tile
    d = desc(n=64, h=34, w=32, c=32, m=16, bits=2)
    kernel, bits = qnn.kernel(d)
    assert (kernel & 0xF, kernel & qnn.KERNEL_ROWS, bits) == (qnn.KERNEL_WINDOW, qnn.KERNEL_ROWS, 8)
    assert qnn.kernel(d, prepared=True) == (qnn.KERNEL_GENERAL, qnn.mma_operand_bits(d))
    assert qnn.tc_kernel(d) == qnn.ALGO_TC_GENERAL


def test_prepared():
    assert qnn.kernel(desc(), prepared=True) == (qnn.KERNEL_WINDOW, 16)
    assert qnn.kernel(desc(c=128, m=128), prepared=True) == (qnn.KERNEL_GATHER, 16)
    for d in (desc(stride=2), desc(algo=qnn.ALGO_DIRECT), desc(bits=1)):
        with pytest.raises(qnn.QnnError) as e:
            qnn.kernel(d, prepared=True)
        assert e.value.status == qnn.QNN_EUNSUPPORTED
    for bad in (desc(bits=5), desc(bits=1, c=12), desc(h=0)):
        with pytest.raises(qnn.QnnError):
            qnn.kernel(bad)


@pytest.mark.parametrize("c,m,k,want", [(128, 8, 1, qnn.KERNEL_COUNT), (128, 40, 1, qnn.KERNEL_COUNT),
                                        (128, 48, 1, qnn.KERNEL_WINDOW), (64, 96, 1, qnn.KERNEL_WINDOW),
                                        (64, 88, 1, qnn.KERNEL_COUNT), (32, 16, 3, qnn.KERNEL_COUNT),
                                        (32, 32, 3, qnn.KERNEL_WINDOW)])
def test_binary_line(c, m, k, want):
    """INT-1 layers run on the window kernel from 6144 products per pixel on."""
    assert qnn.kernel(desc(w=32, c=c, m=m, k=k, pad=k // 2, bits=1))[0] & 0xF == want


@pytest.mark.parametrize("n,h,w,c,m,k,bits,rows", [(2, 34, 28, 24, 112, 3, 8, False), (1, 15, 32, 24, 64, 1, 8, False),
                                                   (5, 26, 44, 40, 16, 1, 8, True), (52, 15, 52, 56, 32, 3, 8, True),
                                                   (2, 29, 32, 32, 64, 3, 2, True)])
def test_whole_rows_line(n, h, w, c, m, k, bits, rows):
    """INT-8 layers of few tiles stay on the general kernel."""
    kernel, _ = qnn.kernel(qnn.conv_desc(n, h, w, c, m, k, k, 1, k // 2, bits))
    assert kernel & ~qnn.KERNEL_STACKED == (qnn.KERNEL_WINDOW | qnn.KERNEL_ROWS if rows else qnn.KERNEL_GENERAL)
