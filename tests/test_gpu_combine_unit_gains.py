"""Backward with unit gains and gain gradients, at head counts around the edges of
what a block's threads hold of a token row (one and two vectors a thread): the
gradients against the 64-bit statement, every output filled with NaN before."""
import numpy as np
import pytest
import torch

from helpers import check_close, np32, seeded

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H,D", [(16, 128), (17, 128), (24, 128), (31, 128), (32, 128), (33, 64), (63, 64), (64, 64), (40, 128)])
def test_every_head_has_its_gradients(H, D):
    from paper_2608_29539_gb300 import logo as L
    T, eps = 37, 1e-6
    x, c, dO = (seeded((T, H, D), H + i).bfloat16() for i in range(3))
    p = torch.sigmoid(seeded((T,), H))
    z, pos, _, row_of, n = L.logo_select(p[None].cuda(), L.LOGO_SELECT_RATIO, ratio=0.4)
    n, sel = int(n), pos[:int(n)].long().cpu()
    nan = lambda *s, dt=torch.bfloat16: torch.full(s, float("nan"), dtype=dt, device="cuda")  # noqa: E731
    f32 = torch.float32
    got = L.logo_combine_bwd_gains(dO[None].cuda(), x[None].cuda(), c.cuda(), p[None].cuda(), z, row_of, eps=eps,
                                   dO_l=nan(1, T, H, D), dO_c=nan(T, H, D), dgate_p=nan(1, T, dt=f32),
                                   dgain_l=nan(H, D, dt=f32), dgain_g=nan(H, D, dt=f32))
    torch.cuda.synchronize()
    w = torch.ones(T, dtype=torch.float64)
    w[sel] -= p[sel].double()

    def grads(x, dy):  # d of x / sqrt(mean x^2 + eps) on dy, and the gain's terms
        r = (x.pow(2).mean(-1, keepdim=True) + eps).rsqrt()
        return r * dy - x * r ** 3 * (x * dy).mean(-1, keepdim=True), dy * x * r, x * r

    d = dO.double()
    dl, gl, yl = grads(x.double(), d * w[:, None, None])
    dc, gc, yc = grads(c[:n].double(), d[sel] * p[sel].double()[:, None, None])
    dp = torch.zeros(T, dtype=torch.float64)
    dp[sel] = (d[sel] * (yc - yl[sel])).sum((1, 2))
    check_close(np32(got[0][0]), dl.numpy(), "dO_l")
    check_close(np32(got[1][:n]), dc.numpy(), "dO_c")
    # fp32 sums of at most H D terms of size a few, relative 2^-24 each
    check_close(np32(got[2][0]), dp.numpy(), "dgate", max_abs=1e-3, rel_l2=1e-5, rel=1e-5)
    check_close(np32(got[3]), gl.sum(0).numpy(), "dgain_l", max_abs=1e-4, rel_l2=1e-5, rel=1e-5)
    check_close(np32(got[4]), gc.sum(0).numpy(), "dgain_g", max_abs=1e-4, rel_l2=1e-5, rel=1e-5)
    assert np.isnan(np32(got[1][n:])).all()
