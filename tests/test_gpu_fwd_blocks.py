"""The forward's hand-over of the running max between the two softmax
warpgroups (even and odd KV blocks): items of one, two and an odd number of
blocks, scores that keep growing along the keys (O is rescaled at nearly every
block, by either warpgroup), rows that see no key of an item's first block."""
import pytest
import torch

import oracle
from helpers import check_close, np32, seeded

pytestmark = pytest.mark.gpu


def _growing(B, T, Hq, Hkv, D, seed, growth):
    """K scaled up along the sequence: row maxima grow by more than 2^8 from block to block."""
    q, k, v = (seeded((B, T, h, D), seed + i, torch.float32) for i, h in enumerate((Hq, Hkv, Hkv)))
    if growth:
        k = k * (0.25 + torch.arange(T) / 96.0)[None, :, None, None]
    return q.bfloat16(), k.bfloat16(), v.bfloat16()


@pytest.mark.parametrize("growth", [False, True])
@pytest.mark.parametrize("B,T,Hq,Hkv,D,W", [
    (2, 100, 2, 1, 128, 40),    # one block an item
    (1, 640, 4, 2, 128, 130),   # one to three blocks: the warpgroups swap parity between items
    (1, 901, 3, 3, 64, 257),    # ragged end, odd head count
    (2, 1024, 2, 2, 64, 1024),  # one to eight blocks
    (1, 515, 2, 2, 128, 128),   # last row of a tile sees nothing of the first block
])
def test_local_blocks(B, T, Hq, Hkv, D, W, growth):
    from paper_2608_29539_gb300 import logo as L
    q, k, v = _growing(B, T, Hq, Hkv, D, 17 * T + W, growth)
    o, lse = L.logo_local_attn_fwd(q.cuda(), k.cuda(), v.cuda(), W)
    torch.cuda.synchronize()
    rb, rt = oracle.local_rows(B, T)
    ro, rl = oracle.attn_fwd(np32(q), np32(k), np32(v), rb, rt, W)
    check_close(np32(o).reshape(B * T, Hq, D), ro, "o")
    check_close(np32(lse).transpose(0, 2, 1).reshape(B * T, Hq), rl, "lse", 1e-3, 1e-5, rel=0.0)


@pytest.mark.parametrize("growth", [False, True])
@pytest.mark.parametrize("B,T,Hq,Hkv,D,ratio", [
    (1, 1500, 4, 2, 64, 0.2),
    (3, 700, 2, 2, 128, 0.5),
    (1, 5000, 2, 1, 128, 0.03),  # split KV ranges
])
def test_global_blocks(B, T, Hq, Hkv, D, ratio, growth):
    from paper_2608_29539_gb300 import logo as L
    q, k, v = _growing(B, T, Hq, Hkv, D, 5 * T + B, growth)
    p = torch.sigmoid(seeded((B, T), T, torch.float32)).contiguous()
    z, pos, cu_q, _, n = L.logo_select(p.cuda(), L.LOGO_SELECT_RATIO, ratio=ratio)
    o_c, lse_c = L.logo_global_sparse_attn_fwd(q.cuda(), k.cuda(), v.cuda(), pos, cu_q, n)
    torch.cuda.synchronize()
    n = int(n)
    rb, rt = oracle.global_rows(pos[:n].cpu().numpy(), cu_q.cpu().numpy())
    ro, rl = oracle.attn_fwd(np32(q), np32(k), np32(v), rb, rt, 0)
    check_close(np32(o_c)[:n], ro, "o_c")
    check_close(np32(lse_c)[:, :n].T, rl, "lse_c", 1e-3, 1e-5, rel=0.0)
