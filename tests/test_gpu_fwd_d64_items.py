"""d = 64 forward with several items a CTA, each of three to eight KV blocks: the
epilogue of an item runs beside the next item's products (two O buffers)."""
import pytest
import torch

import oracle
from helpers import check_close, np32, seeded

pytestmark = pytest.mark.gpu


def _qkv(B, T, Hq, Hkv, seed):
    return [seeded((B, T, h, 64), seed + i, torch.bfloat16) for i, h in enumerate((Hq, Hkv, Hkv))]


@pytest.mark.parametrize("W", [258, 385, 512, 640, 900])
def test_local_items(W):
    from paper_2608_29539_gb300 import logo as L
    B, T, Hq = 4, 1100, 16
    q, k, v = _qkv(B, T, Hq, 4, W)
    dq, dk, dv = q.cuda(), k.cuda(), v.cuda()
    for _ in range(3):
        o, lse = L.logo_local_attn_fwd(dq, dk, dv, W)
    torch.cuda.synchronize()
    assert L.logo_get_device_status() == 0
    rb, rt = oracle.local_rows(B, T)
    ro, rl = oracle.attn_fwd(np32(q), np32(k), np32(v), rb, rt, W)
    check_close(np32(o).reshape(B * T, Hq, 64), ro, "o")
    check_close(np32(lse).transpose(0, 2, 1).reshape(B * T, Hq), rl, "lse", 1e-3, 1e-5, rel=0.0)


@pytest.mark.parametrize("T,ratio", [(640, 0.5), (1000, 0.6), (2500, 0.25)])
def test_global_items(T, ratio):
    from paper_2608_29539_gb300 import logo as L
    B, Hq = 6, 16
    q, k, v = _qkv(B, T, Hq, 8, T)
    p = torch.sigmoid(seeded((B, T), T, torch.float32)).contiguous()
    _, pos, cu_q, _, n = L.logo_select(p.cuda(), L.LOGO_SELECT_RATIO, ratio=ratio)
    o_c, lse_c = L.logo_global_sparse_attn_fwd(q.cuda(), k.cuda(), v.cuda(), pos, cu_q, n)
    torch.cuda.synchronize()
    assert L.logo_get_device_status() == 0
    n = int(n)
    rb, rt = oracle.global_rows(pos[:n].cpu().numpy(), cu_q.cpu().numpy())
    ro, rl = oracle.attn_fwd(np32(q), np32(k), np32(v), rb, rt, 0)
    check_close(np32(o_c)[:n], ro, "o_c")
    check_close(np32(lse_c)[:, :n].T, rl, "lse_c", 1e-3, 1e-5, rel=0.0)
