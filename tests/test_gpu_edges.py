"""Edge sizes of individual kernels: remainders of their tiles, the smallest and the largest of a dispatch rule's
range, each against the oracle or an exact reordering of the input."""
import numpy as np
import pytest

from paper_2604_19654_b200 import build as B
from paper_2604_19654_b200 import feplb as F
from paper_2604_19654_b200 import workloads as W

from gpu_utils import DeviceCase
from test_gpu_parity import _ffn_case

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    B.build()


@pytest.mark.parametrize("E,d,f", [(1, 128, 64), (3, 384, 64), (2, 128, 320), (5, 640, 192)])
def test_transpose_partial_tiles(E, d, f):
    """128 x 128 tiles with a remainder of 64 in either direction, and matrices smaller than one tile."""
    import torch
    case = DeviceCase(W.get_workload("cfg1").with_(E=E, R=1, K=1, T=8, d=d, f=f))
    w1t, w3t = (torch.zeros(E, d, f, dtype=torch.bfloat16, device="cuda") for _ in range(2))
    w2t = torch.zeros(E, f, d, dtype=torch.bfloat16, device="cuda")
    case.ctx.transpose_weights(case.d_w1, case.d_w3, case.d_w2, w1t, w3t, w2t)
    for got, src in ((w1t, case.w1), (w3t, case.w3), (w2t, case.w2)):
        assert np.array_equal(F.bf16_bits(got), src.transpose(0, 2, 1))
    case.close()


@pytest.mark.parametrize("form", [F.FORM_SINGLE, F.FORM_PAIR])
@pytest.mark.parametrize("E,d,f,rows", [
    (2, 128, 64, [1, 130]),            # one narrow N tile in both passes
    (3, 384, 192, [257, 0, 31]),       # a full and a narrow N tile in both passes
    (2, 640, 320, [128, 129]),         # two full and one narrow
    (2, 1920, 704, [90, 300]),         # many of each, the ring wraps
])
def test_expert_ffn_narrow_last_n_tile(E, d, f, rows, form):
    """Widths that are not multiples of the N tile: f % 128 = 64 (pass 1) and d % 256 = 128 (pass 2)."""
    _ffn_case(E, d, f, rows, form=form)
