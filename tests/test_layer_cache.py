"""Sizes that the ABI refuses stay refused once an equal size has been used (no GPU needed)."""
from fractions import Fraction

import numpy as np
import pytest

from paper_1908_11263_gb300 import build as qbuild
from paper_1908_11263_gb300 import qnn


@pytest.fixture(scope="module", autouse=True)
def lib():
    qbuild.build()
    qnn.load()


def _sizes(stride=(1, 1), pad=(1, 1), bits=8, shift=3, algo=qnn.ALGO_AUTO):
    return 2, 16, 16, 32, 64, 3, 3, *stride, *pad, bits, shift, algo


@pytest.mark.parametrize("other", [float, Fraction])
@pytest.mark.parametrize("used_first", [False, True])
def test_values_of_other_types(other, used_first):
    qnn._layer.cache_clear()
    if used_first:
        qnn._layer(*_sizes())
    for kw in (dict(bits=other(8)), dict(shift=other(3)), dict(algo=other(0)), dict(stride=(other(1), 1)),
               dict(pad=(1, other(1)))):
        with pytest.raises(TypeError):
            qnn._layer(*_sizes(**kw))


def test_integers_of_any_type():
    qnn._layer.cache_clear()
    first = qnn._layer(*_sizes())
    assert qnn._layer(*_sizes()) is first
    for kw in (dict(bits=np.int64(8)), dict(stride=(True, 1)), dict(shift=np.int32(3))):
        assert qnn._layer(*_sizes(**kw)).out_shape == first.out_shape
    assert qnn._pair(2) == (2, 2) and qnn._pair([1, 3]) == (1, 3)
    with pytest.raises(ValueError):
        qnn._pair((1, 2, 3))
