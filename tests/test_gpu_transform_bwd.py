"""LP backward at the edges of its tiles: both head dimensions (pairs of 64-wide
heads, an odd one left over), ragged lengths, more tiles than a CTA's two
buffers, selected rows across sequences, none and all of them selected."""
import pytest
import torch

import oracle
from helpers import check_close, np32, seeded

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("accumulate", [False, True])
@pytest.mark.parametrize("B,T,H,D,ratio", [
    (1, 1, 1, 64, None), (2, 130, 3, 64, None), (1, 129, 5, 64, 0.5), (3, 257, 2, 128, None), (3, 300, 4, 128, 0.4),
    (1, 4000, 2, 128, None), (1, 6000, 1, 64, 1.0), (2, 500, 6, 128, 0.0), (1, 9000, 32, 128, 0.1), (1, 700, 64, 128, None),
])
def test_lp_bwd(B, T, H, D, ratio, accumulate):
    from paper_2608_29539_gb300 import logo as L
    s = 7 * T + H
    u, g, d0 = (seeded((B, T, H, D), s + i, torch.bfloat16) for i in range(3))
    a = (torch.eye(D).expand(H, D, D) + 0.05 * seeded((H, D, D), s + 3)).bfloat16().contiguous()
    rows = where = None
    if ratio is not None:
        p = torch.sigmoid(seeded((B, T), s + 4)).contiguous()
        _, pos, cu_q, _, n = L.logo_select(p.cuda(), L.LOGO_SELECT_RATIO, ratio=ratio)
        rows = (pos, cu_q, n)
        where = oracle.global_rows(pos[:int(n)].cpu().numpy(), cu_q.cpu().numpy())
    du = d0.cuda()
    du, da = L.logo_branch_transform_bwd(u.cuda(), g.cuda(), a=a.cuda(), rows=rows, du_l=du, accumulate=accumulate)
    torch.cuda.synchronize()
    live = torch.zeros((B, T), dtype=torch.bool)
    if where is None:
        live[:] = True
    else:
        live[torch.from_numpy(where[0]).long(), torch.from_numpy(where[1]).long()] = True
    gd = g.double() * live[..., None, None]
    share = torch.einsum("bthj,hij->bthi", gd, a.double())
    ref = torch.where(live[..., None, None], share + (d0.double() if accumulate else 0.0), d0.double())
    check_close(np32(du), ref.numpy(), "du")
    # fp32 sums of B*T products: the tensor cores' accumulation, a wide margin
    rda = torch.einsum("bthi,bthj->hij", u.double(), gd)
    check_close(np32(da), rda.numpy(), "dA", 2e-2, 1e-5, rel=1e-4)
