"""The fp32 correlation kernel of grad_w at its edges: widths off the four-pixel quads, one row, one column, channel counts on
and off its tiles, every kernel side with an instance, fewer images than SMs (row bands) and more (several units per CTA)."""
import numpy as np
import pytest

from conftest import nmax_err
from paper_2410_14634_b200 import workloads

pytestmark = pytest.mark.gpu

SHAPES = [(1, 5, 7, 9, 3), (2, 6, 1, 13, 3), (3, 7, 11, 1, 2), (2, 4, 33, 30, 5), (1, 8, 64, 62, 2), (300, 9, 5, 6, 3), (4, 12, 16, 16, 5), (2, 13, 9, 7, 3),
          (3, 24, 10, 11, 3), (2, 3, 40, 37, 7), (2, 2, 21, 24, 9), (2, 4, 26, 26, 11), (1, 3, 12, 130, 11), (5, 40, 6, 5, 4), (2, 5, 8, 8, 1)]


@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "x".join(map(str, s)))
def test_grad_w_fp32_matches_oracle(shape):
    import torch
    from oracle import api as oracle
    from paper_2410_14634_b200 import binding as B
    Bn, C, H, W, k = shape
    w, y, gx = workloads.make_custom(77 + sum(shape), Bn, C, H, W, k, sigma=0.15 / np.sqrt(C * k * k))
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    prev = B.invconv_set_option(B.OPT_GRADW_TENSOR_PIPE, 0), B.invconv_set_option(B.OPT_GRADW_SEPARATE, 1)
    try:
        x = B.invconv_forward(dev(y), dev(w))
        gy, gw = B.invconv_backward(dev(gx), x, dev(w))
        gw2 = B.invconv_backward(dev(gx), x, dev(w))[1]
        torch.cuda.synchronize()
        assert B.invconv_get_status() == 0
    finally:
        B.invconv_set_option(B.OPT_GRADW_TENSOR_PIPE, prev[0])
        B.invconv_set_option(B.OPT_GRADW_SEPARATE, prev[1])
    ref = oracle.invconv_grad_w(gy.cpu().numpy(), x.cpu().numpy(), k)
    assert nmax_err(gw.cpu().numpy(), ref) <= 5e-6
    assert torch.equal(gw, gw2)
