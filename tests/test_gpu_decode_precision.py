"""Rounding of the decode kernel's probabilities.  A warp takes 16 adjacent
cache rows of a sub-tile at a time; the largest probability among them is a
power of two relative to what its sums are kept against, so bf16 holds it
exactly.  With one visible key in every 16 rows nothing is left but the rounding
of the output: |o - ref| <= 2^-8 |ref| (half an ulp of bf16), plus 2^-14 of the
weighted |v|, 64 times what a score's fp32 accumulation and the exponential's
2^-22 move a weight by (two of them, scores below 32 in log2 units)."""
import numpy as np
import pytest
import torch

from helpers import BF16_ROUNDING, np32

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ring,B,R,Hq,Hkv,D", [
    (False, 1, 8192, 4, 1, 128),   # one pair in short runs
    (False, 160, 1024, 2, 2, 128), # longer runs, cut inside pairs
    (True, 150, 1024, 8, 4, 64),   # whole pairs of 16 sub-tiles
    (True, 3, 640, 16, 1, 64),
])
def test_decode_largest_probability_is_exact(ring, B, R, Hq, Hkv, D):
    from paper_2608_29539_gb300 import logo as G
    g = torch.Generator().manual_seed(R + B)
    q = torch.zeros((B, Hq, D))
    q[..., 0] = 1.0 + torch.rand((B, Hq), generator=g)
    k = torch.zeros((B, R, Hkv, D))
    k[..., 0] = -200.0                                                    # no weight at all
    k[:, ::16, :, 0] = 8.0 * torch.rand((B, (R + 15) // 16, Hkv), generator=g)  # one key of 16 rows
    v = torch.randn((B, R, Hkv, D), generator=g)
    q, k, v = (t.bfloat16() for t in (q, k, v))
    n = torch.full((B,), R, dtype=torch.int32, device="cuda")
    if ring:
        o = G.logo_decode_local_attn(q.cuda(), k.cuda(), v.cuda(), n, R, scale=1.0)
    else:
        cu_q = torch.arange(B + 1, dtype=torch.int32, device="cuda")
        o = G.logo_decode_global_sparse_attn(q.cuda(), k.cuda(), v.cuda(), n, cu_q, cu_q[-1:], scale=1.0)
    s = (q[..., :1].double() * k[..., 0].double().permute(0, 2, 1).repeat_interleave(Hq // Hkv, 1))  # [B, Hq, R]
    w = torch.softmax(s, -1)
    vv = v.double().repeat_interleave(Hq // Hkv, 2)
    ref = torch.einsum("bhr,brhd->bhd", w, vv).numpy()
    mass = torch.einsum("bhr,brhd->bhd", w, vv.abs()).numpy()
    used = np.abs(np32(o) - ref) / (BF16_ROUNDING * np.abs(ref) + 2.0 ** -14 * mass)
    assert used.max() <= 1.0, used.max()
