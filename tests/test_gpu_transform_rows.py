"""LP forward on selected rows at the edges of its 128-row tiles: both head
dimensions, none, one, a tile more or less, rows across sequences, more tiles
than a CTA's two buffers; rows that are not selected keep what they held."""
import pytest
import torch

from helpers import check_close, np32, seeded

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,T,H,D,n", [
    (1, 40, 1, 64, 0), (1, 40, 2, 128, 1), (2, 200, 3, 64, 127), (1, 300, 4, 128, 128), (3, 150, 5, 128, 129),
    (2, 900, 2, 64, 1301), (1, 5000, 64, 128, 4700), (1, 2500, 40, 64, 2500),
])
def test_lp_fwd_rows(B, T, H, D, n):
    from paper_2608_29539_gb300 import logo as L
    u, keep = (seeded((B, T, H, D), T + i, torch.bfloat16) for i in range(2))
    a = (torch.eye(D).expand(H, D, D) + 0.05 * seeded((H, D, D), T + 3)).bfloat16().contiguous()
    p = torch.zeros(B * T)
    p[torch.randperm(B * T, generator=torch.Generator().manual_seed(T))[:n]] = 1.0
    _, pos, cu_q, _, m = L.logo_select(p.view(B, T).cuda(), L.LOGO_SELECT_THRESHOLD, b_th=0.5)
    assert int(m) == n
    out = keep.cuda()
    L.logo_branch_transform(u.cuda(), rows=(pos, cu_q, m), a=a.cuda(), u_g=out)
    torch.cuda.synchronize()
    ref = torch.where((p > 0).view(B, T, 1, 1), torch.einsum("bthi,hij->bthj", u.double(), a.double()), keep.double())
    check_close(np32(out), ref.numpy(), "u_g")
