"""Global forward with few, long tiles on either side of the length from which
KV ranges may be split (32 blocks of 128 keys: 8 a share and a gain of 24): what is split is merged, and
what cannot be is not left unmerged."""
import pytest
import torch

import oracle
from helpers import check_close, np32, seeded

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("D", [64, 128])
@pytest.mark.parametrize("T", [3968, 3969, 4096, 4225])
def test_global_fwd_around_split_length(T, D):
    from paper_2608_29539_gb300 import logo as L
    q, k, v = (seeded((1, T, 1, D), T + i, torch.bfloat16) for i in range(3))
    p = torch.zeros((1, T))
    p[0, -5:] = 1.0   # one tile that sees every block
    p[0, 3] = 1.0
    _, pos, cu_q, _, n = L.logo_select(p.cuda(), L.LOGO_SELECT_THRESHOLD, b_th=0.5)
    o_c, lse_c = L.logo_global_sparse_attn_fwd(q.cuda(), k.cuda(), v.cuda(), pos, cu_q, n)
    torch.cuda.synchronize()
    rb, rt = oracle.global_rows(pos[:6].cpu().numpy(), cu_q.cpu().numpy())
    ro, rl = oracle.attn_fwd(np32(q), np32(k), np32(v), rb, rt, 0)
    check_close(np32(o_c)[:6], ro, "o_c")
    check_close(np32(lse_c)[:, :6].T, rl, "lse_c", 1e-3, 1e-5, rel=0.0)
