"""dA of the LP backward written into a larger fp32 buffer, at offsets that are
multiples of 4 bytes only: the same bits as in a buffer of its own, and nothing
beside them."""
import pytest
import torch

from helpers import seeded

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,T,H,D,select", [(1, 300, 3, 64, False), (2, 257, 2, 128, False), (2, 257, 2, 128, True)])
def test_da_at_any_float(B, T, H, D, select):
    from paper_2608_29539_gb300 import logo as L
    u, g = (seeded((B, T, H, D), T + i, torch.bfloat16).cuda() for i in range(2))
    a = seeded((H, D, D), T + 2).bfloat16().contiguous().cuda()
    rows = (None,) * 3
    if select:
        _, pos, cu_q, _, n = L.logo_select(torch.sigmoid(seeded((B, T), 3)).cuda(), L.LOGO_SELECT_RATIO, ratio=0.3)
        rows = (pos, cu_q, n)
    du, ref = L.logo_branch_transform_bwd(u, g, a=a, rows=rows if select else None)
    d = L.Dims(B, T, H, H, D)
    ws = torch.empty(L.lib().logo_branch_transform_bwd_workspace_size(d), dtype=torch.uint8, device="cuda")
    for off in (1, 2, 3, 4):
        flat = torch.full((H * D * D + 8,), 7.0, device="cuda")
        assert flat.data_ptr() % 16 == 0
        L._call("logo_branch_transform_bwd", L._p(u), L._p(a), None, *(L._p(t) for t in rows), L._p(g), L._p(du), 0,
                flat.data_ptr() + 4 * off, None, None, d, L._p(ws), ws.numel(), L._stream())
        torch.cuda.synchronize()
        assert torch.equal(flat[off:off + H * D * D], ref.flatten())
        assert bool((flat[:off] == 7.0).all()) and bool((flat[off + H * D * D:] == 7.0).all())
