"""The d = 64 local backward of short and odd sequences, whose rows' statistics
end inside a tile of 128: many of them, in a workspace that held NaN."""
import pytest
import torch

import oracle
from helpers import check_close, np32, seeded

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,T,Hq,Hkv,W", [(300, 1, 3, 1, 1), (200, 2, 2, 2, 2), (150, 3, 4, 2, 2), (40, 63, 2, 1, 20),
                                          (9, 127, 3, 3, 200), (6, 257, 4, 2, 130), (2, 4095, 2, 1, 1000)])
def test_short_sequences(B, T, Hq, Hkv, W):
    from paper_2608_29539_gb300 import logo as L
    q, k, v, dO = [seeded((B, T, h, 64), B + i, torch.bfloat16) for i, h in enumerate((Hq, Hkv, Hkv, Hq))]
    qc, kc, vc, dc = q.cuda(), k.cuda(), v.cuda(), dO.cuda()
    o, lse = L.logo_local_attn_fwd(qc, kc, vc, W)
    ws = torch.full((L.workspace_bytes("local_bwd", L.dims_of(q, k)),), 255, dtype=torch.uint8, device="cuda")
    dq, dk, dv = L.logo_local_attn_bwd(qc, kc, vc, o, lse, dc, W, workspace=ws)
    torch.cuda.synchronize()
    rb, rt = oracle.local_rows(B, T)
    rdq, rdk, rdv = oracle.attn_bwd(np32(q), np32(k), np32(v), rb, rt, W, np32(dO).reshape(B * T, Hq, 64))
    check_close(np32(dq).reshape(B * T, Hq, 64), rdq, "dq")
    check_close(np32(dk), rdk, "dk")
    check_close(np32(dv), rdv, "dv")
