"""The window kernel's fused 2x2 max-pool, whose lanes exchange strips and words (store_pooled), byte for byte against
the oracle's two layers in sequence: filter counts at the edges of a lane's word and of an 8-channel block, one and two
strips, partial strips, folded kernel columns."""
import numpy as np
import pytest
import torch

from paper_1908_11263_gb300 import qnn

from gpu_util import first_mismatch
from test_gpu_conv_pool import run_fused, run_oracle, spread_case

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def loaded():
    qnn.load(build_if_missing=True)
    torch.cuda.set_device(0)


# (n, h, w, c, k, pad, bits): two strips; one; a second strip with one pooled column; folded 5 x 5 and 3 x 3
GEOMETRY = [
    (2, 18, 16, 32, 3, 1, 0),
    (3, 8, 8, 32, 5, 2, 0),
    (1, 11, 14, 32, 3, 0, 0),
    (2, 17, 32, 3, 5, 2, 8),
    (1, 34, 16, 3, 3, 1, 8),
]
FILTERS = {8: (1, 3, 4, 5, 12, 33, 64), 4: (2, 6, 8, 34, 72), 2: (4, 8, 12, 36, 128)}


@pytest.mark.parametrize("geometry", GEOMETRY, ids=lambda s: "x".join(str(v) for v in s))
@pytest.mark.parametrize("bits", [8, 4, 2])
def test_pool_exchange(geometry, bits):
    n, h, w, c, k, pad, only = geometry
    if only not in (0, bits):
        pytest.skip("folded layers are INT-8")
    for m in FILTERS[bits]:
        case = spread_case(m + sum(geometry), n, h, w, c, m, k, bits, m % 2 == 1)
        out, _ = run_fused(*case, bits, pad, qnn.ALGO_TC_WINDOW)
        want = run_oracle(*case, bits, pad)
        assert first_mismatch(out.cpu().numpy().reshape(-1), want) is None, m
