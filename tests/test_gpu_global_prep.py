"""The packed query rows of the global forward at the edges of the kernel that
gathers them (four rows a block) beside the schedule: no row, a few, a block
more or less, sequences without any, rows wider than a block's quarter."""
import pytest
import torch

import oracle
from helpers import check_close, np32, seeded

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,T,Hq,Hkv,D,counts", [
    (1, 40, 1, 1, 64, [0]), (1, 40, 1, 1, 64, [1]), (2, 50, 2, 1, 128, [0, 3]), (3, 60, 3, 3, 64, [4, 0, 5]),
    (2, 300, 4, 2, 128, [127, 130]), (1, 700, 32, 8, 128, [609]), (1, 400, 48, 4, 128, [301]),
])
def test_global_fwd_rows(B, T, Hq, Hkv, D, counts):
    from paper_2608_29539_gb300 import logo as L
    q, k, v = (seeded((B, T, h, D), T + i, torch.bfloat16) for i, h in enumerate((Hq, Hkv, Hkv)))
    p = torch.zeros((B, T))
    for b, c in enumerate(counts):
        p[b, torch.randperm(T, generator=torch.Generator().manual_seed(T + b))[:c]] = 1.0
    _, pos, cu_q, _, n = L.logo_select(p.cuda(), L.LOGO_SELECT_THRESHOLD, b_th=0.5)
    o_c, lse_c = L.logo_global_sparse_attn_fwd(q.cuda(), k.cuda(), v.cuda(), pos, cu_q, n)
    torch.cuda.synchronize()
    n = int(n)
    assert n == sum(counts)
    if n == 0:
        return
    rb, rt = oracle.global_rows(pos[:n].cpu().numpy(), cu_q.cpu().numpy())
    ro, rl = oracle.attn_fwd(np32(q), np32(k), np32(v), rb, rt, 0)
    check_close(np32(o_c)[:n], ro, "o_c")
    check_close(np32(lse_c)[:, :n].T, rl, "lse_c", 1e-3, 1e-5, rel=0.0)
