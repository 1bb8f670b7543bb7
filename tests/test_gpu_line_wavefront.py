"""The line wavefront (one thread per image row and output channel) at the sizes where it can go wrong: every kernel side and
channel count at the edges of its instances, widths off and on the 4-column pieces, images of one row or column, bands with halo
rows, several images per CTA, both storage types, the flow step's fused neighbours."""
import numpy as np
import pytest

from conftest import nmax_err
from paper_2410_14634_b200 import workloads

pytestmark = pytest.mark.gpu

SHAPES = [
    (3, 1, 5, 7, 2), (2, 2, 33, 40, 3), (300, 2, 9, 6, 3), (3, 3, 64, 64, 5), (2, 3, 70, 9, 5), (2, 4, 130, 60, 5), (9, 4, 70, 132, 5), (3, 3, 256, 64, 3), (2, 3, 210, 50, 3), (2, 12, 52, 36, 2), (3, 4, 64, 60, 11), (1, 4, 1, 33, 3),
    (2, 4, 40, 1, 5), (5, 5, 7, 9, 3), (3, 6, 45, 51, 3), (2, 8, 31, 17, 2), (160, 8, 16, 16, 3), (2, 9, 13, 12, 5), (301, 12, 4, 5, 3),
    (3, 12, 36, 36, 3), (2, 12, 32, 32, 5), (4, 13, 12, 10, 3), (3, 16, 32, 30, 3), (2, 16, 9, 8, 2), (2, 1, 40, 36, 7), (2, 2, 20, 18, 9),
    (3, 3, 64, 48, 7), (2, 4, 42, 40, 9), (2, 3, 32, 32, 11), (2, 4, 50, 13, 11), (1, 1, 12, 8, 11),
]


@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "x".join(map(str, s)))
def test_line_wavefront_matches_oracle(shape):
    import torch
    from oracle import api as oracle, flow_step
    from paper_2410_14634_b200 import binding as B
    Bn, C, H, W, k = shape
    sigma = 0.15 / np.sqrt(C * k * k)
    w, y, gx = workloads.make_custom(31 + sum(shape), Bn, C, H, W, k, sigma=sigma, masked_fill=np.nan)
    rng = np.random.default_rng(2)
    s, b = rng.uniform(0.5, 1.5, C).astype(np.float32), rng.normal(0, 0.3, C).astype(np.float32)
    V = np.linalg.qr(rng.normal(size=(C, C)))[0].astype(np.float32)
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    off = lambda a: torch.cat([torch.zeros(1), torch.from_numpy(a).reshape(-1)]).cuda()[1:].view(a.shape)     # 4 bytes off
    prev = B.invconv_set_option(B.OPT_LINE, 1)
    try:
        wd = dev(w)
        x, ld = B.invconv_forward_logdet(dev(y), wd)
        x_off = B.invconv_forward(off(y), wd)
        gy, _ = B.invconv_backward(dev(gx), x, wd, need_grad_w=False)
        gy_off, _ = B.invconv_backward(off(gx), x, wd, need_grad_w=False)
        y16 = dev(y).to(torch.bfloat16)
        x16 = B.invconv_forward_bf16(y16, wd)
        x2, u, _ = B.invconv_flow_step_forward(dev(y), wd, dev(s), dev(b), dev(V))
        gy2 = B.invconv_flow_step_backward(dev(gx), x2, wd, dev(s), dev(b), dev(V))[0]
        torch.cuda.synchronize()
        assert B.invconv_get_status() == 0
    finally:
        B.invconv_set_option(B.OPT_LINE, prev)
    x_ref = oracle.invconv_forward(y, w)
    gy_ref = oracle.invconv_grad_y(gx, w)
    assert nmax_err(x.cpu().numpy(), x_ref) <= 2e-6 and nmax_err(gy.cpu().numpy(), gy_ref) <= 2e-6
    assert torch.equal(x, x_off) and torch.equal(gy, gy_off) and torch.equal(x, x2)
    assert abs(float(ld) - oracle.logdet(w, H, W)) <= 1e-5 * max(abs(oracle.logdet(w, H, W)), H * W * 1e-3)
    ref16 = oracle.invconv_forward(y16.float().cpu().numpy(), w)
    assert nmax_err(x16.float().cpu().numpy(), ref16) <= 5e-3
    u_ref = flow_step.step_forward(y, w, s, b, V)[1]
    assert nmax_err(u.cpu().numpy(), u_ref) <= 5e-6
    gy2_ref = oracle.invconv_grad_y((np.einsum("oc,nohw->nchw", V.astype(np.float64), gx.astype(np.float64)) * s[None, :, None, None]).astype(np.float32), w)
    assert nmax_err(gy2.cpu().numpy(), gy2_ref) <= 5e-6
