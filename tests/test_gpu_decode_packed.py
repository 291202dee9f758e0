"""The global decode call on short caches, where a CTA takes whole pairs of the
packed rows: none, one, some and all of the sequences selected, several pairs a
CTA, and empty caches among the selected."""
import numpy as np
import pytest
import torch

from helpers import check_close, np32, seeded

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,R,Hq,Hkv,D", [(400, 128, 2, 2, 64), (41, 448, 8, 8, 64), (7, 200, 16, 1, 128)])
@pytest.mark.parametrize("every", [0, 1, 3, 1000])
def test_packed_rows(B, R, Hq, Hkv, D, every):
    from paper_2608_29539_gb300 import logo as G
    q, k, v = (seeded(s, B + i).bfloat16() for i, s in enumerate([(B, Hq, D)] + 2 * [(B, R, Hkv, D)]))
    n = 1 + torch.arange(B) * 37 % R
    n[B // 2] = 0
    sel = (torch.arange(B) % every == every - 1) if 0 < every < 1000 else torch.zeros(B, dtype=torch.bool)
    if every == 1000:
        sel[B - 1] = True
    cu_q = torch.cat([torch.zeros(1), sel.cumsum(0)]).int()
    o = torch.full((B, Hq, D), 9.0, dtype=torch.bfloat16).cuda()
    G.logo_decode_global_sparse_attn(q.cuda(), k.cuda(), v.cuda(), n.int().cuda(), cu_q.cuda(), cu_q[-1:].cuda(), o_c=o)
    torch.cuda.synchronize()
    rows = sel.nonzero()[:, 0]
    keep = n[rows] > 0  # a selected empty cache has no row to write
    rep = Hq // Hkv
    kk, vv = (t[rows].double().repeat_interleave(rep, 2) for t in (k, v))
    s = torch.einsum("bhd,bjhd->bhj", q[rows].double(), kk) / D ** 0.5
    s.masked_fill_((torch.arange(R)[None, :] >= n[rows, None])[:, None], float("-inf"))
    ref = torch.einsum("bhj,bjhd->bhd", torch.softmax(s, -1), vv)
    got = np32(o)
    check_close(got[:len(rows)][keep.numpy()], ref[keep].numpy(), "o")
    assert (got[len(rows):] == 9.0).all()
