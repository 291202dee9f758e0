"""The d = 128 backward at the edges of its 64-row query tiles and 128-key
blocks: ragged ends, windows smaller and larger than a tile, grouped heads,
tiles that hold rows of two sequences, blocks no selected row sees, CTAs with
many one-tile items."""
import pytest
import torch

import oracle
from helpers import check_close, np32, seeded

pytestmark = pytest.mark.gpu


def _qkvd(B, T, Hq, Hkv, seed):
    return [seeded((B, T, h, 128), seed + i, torch.bfloat16) for i, h in enumerate((Hq, Hkv, Hkv, Hq))]


@pytest.mark.parametrize("B,T,Hq,Hkv,W", [(3, 333, 4, 2, 50), (1, 1030, 6, 2, 257), (2, 128, 2, 2, 128), (1, 129, 1, 1, 1),
                                          (2, 1300, 8, 1, 1300), (5, 31, 2, 2, 7), (64, 65, 8, 8, 20)])
def test_local_bwd128(B, T, Hq, Hkv, W):
    from paper_2608_29539_gb300 import logo as L
    q, k, v, dO = _qkvd(B, T, Hq, Hkv, T + W)
    qc, kc, vc, dc = q.cuda(), k.cuda(), v.cuda(), dO.cuda()
    o, lse = L.logo_local_attn_fwd(qc, kc, vc, W)
    dq, dk, dv = L.logo_local_attn_bwd(qc, kc, vc, o, lse, dc, W)
    torch.cuda.synchronize()
    rb, rt = oracle.local_rows(B, T)
    rdq, rdk, rdv = oracle.attn_bwd(np32(q), np32(k), np32(v), rb, rt, W, np32(dO).reshape(B * T, Hq, 128))
    check_close(np32(dq).reshape(B * T, Hq, 128), rdq, "dq")
    check_close(np32(dk), rdk, "dk")
    check_close(np32(dv), rdv, "dv")


@pytest.mark.parametrize("B,T,Hq,Hkv,chosen", [
    (3, 257, 4, 2, 0.5), (1, 300, 2, 2, 1.0), (2, 400, 2, 2, 0.0), (4, 515, 6, 3, 0.1),
    (48, 130, 4, 4, 0.05), (1, 1500, 4, 1, "first"),  # later blocks are seen by no selected row
])
def test_global_bwd128(B, T, Hq, Hkv, chosen):
    from paper_2608_29539_gb300 import logo as L
    q, k, v, _ = _qkvd(B, T, Hq, Hkv, 3 * T + B)
    dO_c = seeded((B * T, Hq, 128), T, torch.bfloat16)
    if chosen == "first":
        p, ratio = (torch.arange(T) < 200).float()[None].repeat(B, 1).contiguous(), 200.5 / T
    else:
        p, ratio = torch.sigmoid(seeded((B, T), T + 1)).contiguous(), chosen
    z, pos, cu_q, _, n = L.logo_select(p.cuda(), L.LOGO_SELECT_RATIO, ratio=ratio)
    qc, kc, vc = q.cuda(), k.cuda(), v.cuda()
    o_c, lse_c = L.logo_global_sparse_attn_fwd(qc, kc, vc, pos, cu_q, n)
    dq, dk, dv = L.logo_global_sparse_attn_bwd(qc, kc, vc, pos, cu_q, n, o_c, lse_c, dO_c.cuda())
    torch.cuda.synchronize()
    n = int(n)
    rb, rt = oracle.global_rows(pos[:n].cpu().numpy(), cu_q.cpu().numpy())
    rdq, rdk, rdv = oracle.attn_bwd(np32(q), np32(k), np32(v), rb, rt, 0, np32(dO_c)[:n])
    full = torch.zeros((B, T, Hq, 128), dtype=torch.float64)
    full[torch.from_numpy(rb).long(), torch.from_numpy(rt).long()] = torch.from_numpy(rdq)
    check_close(np32(dq), full.numpy(), "dq")
    check_close(np32(dk), rdk, "dk")
    check_close(np32(dv), rdv, "dv")
