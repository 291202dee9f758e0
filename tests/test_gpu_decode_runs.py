"""Decoding over equal runs of sub-tiles: sequences of very different lengths,
runs that begin and end inside pairs, pairs cut into many pieces, more than
128 sequences (two rounds of the scan), selections of one and of all."""
import numpy as np
import pytest
import torch

import oracle
from helpers import check_close, np32, seeded

pytestmark = pytest.mark.gpu


def _ref(q, k, v, lens, rows, window):
    B, Hq, D = q.shape
    qf = np.zeros((B, k.shape[1], Hq, D), dtype=np.float32)
    for b in rows:
        qf[b, lens[b] - 1] = np32(q[b])
    o, _ = oracle.attn_fwd(qf, np32(k), np32(v), np.array(rows, np.int32),
                           np.array([lens[b] - 1 for b in rows], np.int32), window)
    return o


@pytest.mark.parametrize("B,L,Hq,Hkv,D,every", [
    (3, 9000, 4, 2, 128, 1),     # a few pairs in many pieces
    (7, 700, 6, 3, 64, 2),
    (200, 130, 2, 1, 64, 3),     # two rounds of the scan, pairs of one to three sub-tiles
    (1, 8192, 1, 1, 128, 1),     # one pair: as many pieces as the merge takes
    (40, 2000, 16, 1, 64, 7),
])
def test_decode_global_runs(B, L, Hq, Hkv, D, every):
    from paper_2608_29539_gb300 import logo as G
    q = seeded((B, Hq, D), B + L, torch.bfloat16)
    k, v = (seeded((B, L, Hkv, D), B + L + i, torch.bfloat16) for i in (1, 2))
    g = torch.Generator().manual_seed(L)
    lens = (torch.rand(B, generator=g) ** 3 * L).long().clamp_(1, L)
    lens[0] = L
    p = torch.zeros((B, 1))
    p[::every] = 0.9
    rows = [b for b in range(B) if p[b, 0] > 0.5]
    for b in range(B):  # rows past the end, and whole unselected caches, are never used
        k[b, lens[b]:] = float("nan")
        v[b, lens[b]:] = float("nan")
    _, _, cu_q, _, n = G.logo_select(p.cuda(), G.LOGO_SELECT_THRESHOLD, b_th=0.5)
    o = torch.full((B, Hq, D), 5.0, dtype=torch.bfloat16, device="cuda")
    for _ in range(2):  # a second call on the same workspace-sized allocations
        G.logo_decode_global_sparse_attn(q.cuda(), k.cuda(), v.cuda(), lens.int().cuda(), cu_q, n, o_c=o)
    torch.cuda.synchronize()
    kk, vv = torch.nan_to_num(k.float()).bfloat16(), torch.nan_to_num(v.float()).bfloat16()
    check_close(np32(o)[:len(rows)], _ref(q, kk, vv, lens.tolist(), rows, 0), "decode global runs")
    assert bool((o[len(rows):] == 5.0).all())


@pytest.mark.parametrize("B,R,W,Hq,Hkv,D", [(2, 4096, 4000, 4, 1, 128), (150, 64, 50, 2, 2, 64), (5, 1024, 777, 8, 8, 128),
                                            (1, 20000, 20000, 2, 1, 64)])
def test_decode_local_runs(B, R, W, Hq, Hkv, D):
    from paper_2608_29539_gb300 import logo as G
    L = 2 * R + 17
    q = seeded((B, Hq, D), B + R, torch.bfloat16)
    k, v = (seeded((B, L, Hkv, D), B + R + i, torch.bfloat16) for i in (1, 2))
    g = torch.Generator().manual_seed(R)
    lens = torch.randint(1, L + 1, (B,), generator=g).tolist()
    kr, vr = (torch.full((B, R, Hkv, D), float("nan"), dtype=torch.bfloat16) for _ in range(2))
    for b, n in enumerate(lens):
        s = torch.arange(max(0, n - min(R, W)), n)
        kr[b, s % R], vr[b, s % R] = k[b, s], v[b, s]
    o = G.logo_decode_local_attn(q.cuda(), kr.cuda(), vr.cuda(), torch.tensor(lens, dtype=torch.int32).cuda(), W)
    torch.cuda.synchronize()
    check_close(np32(o), _ref(q, k, v, lens, list(range(B)), W), "decode local runs")
