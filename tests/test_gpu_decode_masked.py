"""Decode over caches whose masked rows hold keys of bf16's lowest value (a finite
score far below all others), in whole 16-row groups and mixed with others, before
and after the rows that count, whose scores are hundreds of octaves above 1."""
import numpy as np
import pytest
import torch

from helpers import check_close, np32, seeded

pytestmark = pytest.mark.gpu

LOWEST = torch.finfo(torch.bfloat16).min


@pytest.mark.parametrize("ring", [False, True])
@pytest.mark.parametrize("B,R,Hq,Hkv,D,keep", [
    (3, 1000, 4, 2, 64, lambda j: (j // 16) % 2 == 0),   # every second group of 16
    (2, 4096, 8, 1, 128, lambda j: (j // 64) % 3 == 1),  # whole sub-tiles
    (160, 700, 2, 2, 64, lambda j: j % 5 == 2),
    (1, 1500, 16, 1, 128, lambda j: j >= 1400),
])
def test_lowest_value_keys(ring, B, R, Hq, Hkv, D, keep):
    from paper_2608_29539_gb300 import logo as G
    q = torch.zeros((B, Hq, D))
    q[..., 0] = 1.0
    q[..., 1:] = 0.1 * seeded((B, Hq, D - 1), R)
    k = seeded((B, R, Hkv, D), R + 1)
    k[..., 0] = 400.0  # scores of about 200
    seen = keep(torch.arange(R))
    k[:, ~seen] = 0.0
    k[:, ~seen, :, 0] = LOWEST  # scores of about -1.7e38
    v = seeded((B, R, Hkv, D), R + 2)
    q, k, v = (t.bfloat16() for t in (q, k, v))
    n = torch.full((B,), R, dtype=torch.int32, device="cuda")
    if ring:
        o = G.logo_decode_local_attn(q.cuda(), k.cuda(), v.cuda(), n, R, scale=0.5)
    else:
        cu_q = torch.arange(B + 1, dtype=torch.int32, device="cuda")
        o = G.logo_decode_global_sparse_attn(q.cuda(), k.cuda(), v.cuda(), n, cu_q, cu_q[-1:], scale=0.5)
    rep = Hq // Hkv
    s = 0.5 * torch.einsum("bhd,bjhd->bhj", q.double(), k.double().repeat_interleave(rep, 2))
    ref = torch.einsum("bhj,bjhd->bhd", torch.softmax(s, -1), v.double().repeat_interleave(rep, 2))
    assert np.isfinite(np32(o)).all()
    check_close(np32(o), ref.numpy(), "o")
