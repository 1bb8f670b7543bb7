"""The tensor-core wavefront with three-term products at the edges of its range: padded channel counts, every cluster size,
images of one row and of 32 rows, slices on and off 16 bytes, several groups per cluster, groups cut by the shared memory; its
error against a float64 residual is that of an fp32 kernel."""
import numpy as np
import pytest

from conftest import nmax_err
from paper_2410_14634_b200 import workloads

pytestmark = pytest.mark.gpu

SHAPES = [
    (3, 17, 9, 8, 3), (130, 24, 5, 5, 3), (2, 24, 32, 16, 2), (5, 32, 1, 41, 3), (3, 33, 12, 10, 5), (300, 40, 4, 5, 3), (2, 48, 9, 9, 5),
    (9, 56, 7, 6, 2), (2, 64, 9, 9, 3), (4, 66, 3, 31, 3), (3, 80, 6, 7, 2), (2, 81, 5, 9, 3), (40, 96, 6, 4, 3), (2, 96, 13, 11, 2),
    (2, 20, 31, 20, 5),
]


@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "x".join(map(str, s)))
def test_three_term_wavefront_matches_oracle(shape):
    import torch
    from oracle import api as oracle
    from paper_2410_14634_b200 import binding as B
    Bn, C, H, W, k = shape
    w, y, gx = workloads.make_custom(41 + sum(shape), Bn, C, H, W, k, sigma=0.15 / np.sqrt(C * k * k), masked_fill=np.nan)
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    off = lambda a: torch.cat([torch.zeros(1), torch.from_numpy(a).reshape(-1)]).cuda()[1:].view(a.shape)     # 4 bytes off
    wd = dev(w)
    x, ld = B.invconv_forward_logdet(dev(y), wd)
    assert torch.equal(x, B.invconv_forward(off(y), wd))
    gy, gw = B.invconv_backward(dev(gx), x, wd)
    torch.cuda.synchronize()
    assert B.invconv_get_status() == 0
    assert nmax_err(x.cpu().numpy(), oracle.invconv_forward(y, w)) <= 2e-6
    assert nmax_err(gy.cpu().numpy(), oracle.invconv_grad_y(gx, w)) <= 2e-6
    assert abs(float(ld) - oracle.logdet(w, H, W)) <= 1e-5 * max(abs(oracle.logdet(w, H, W)), H * W * 1e-3)
    m = torch.nan_to_num(wd.double())
    m[:, :, k - 1, k - 1] = torch.tril(m[:, :, k - 1, k - 1])
    fx = torch.nn.functional.conv2d(torch.nn.functional.pad(x.double(), (k - 1, 0, k - 1, 0)), m)
    yd = dev(y).double()
    assert (fx - yd).norm() <= 4e-7 * yd.norm()
