"""Gain gradients of a dO column that is infinite: the sum over tokens is infinite
there and finite elsewhere, also where the last tokens leave some of a block's
rows of threads without one."""
import pytest
import torch

from helpers import seeded

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T,H,D", [(50003, 1, 64), (40001, 3, 64), (30007, 1, 128), (9, 1, 64)])
def test_infinite_column(T, H, D):
    from paper_2608_29539_gb300 import logo as L
    o_l, o_c, dO = (seeded((1, T, H, D), T + i).bfloat16() for i in range(3))
    o_l[..., 5], o_c[..., 5], dO[..., 5] = 0.5, 0.25, float("inf")
    p = torch.sigmoid(seeded((1, T), T)).cuda()
    z, _, _, row_of, n = L.logo_select(p, L.LOGO_SELECT_RATIO, ratio=0.5)
    gain = 1.0 + 0.1 * seeded((H, D), T).cuda()
    dgl, dgg = L.logo_combine_bwd_gains(dO.cuda(), o_l.cuda(), o_c.view(T, H, D).cuda(), p, z, row_of, gain, gain)[3:]
    torch.cuda.synchronize()
    inf = torch.zeros((H, D), dtype=torch.bool)
    inf[:, 5] = True
    for g in (dgl, dgg):
        assert torch.equal(g.cpu() == float("inf"), inf) and bool(torch.isfinite(g.cpu()[~inf]).all())
