"""Decode calls with as many (sequence, KV head) pairs as CTAs, on both sides of
the length from which pairs are always cut: a few sequences selected or long, the
others unselected, short or empty."""
import numpy as np
import pytest
import torch

import oracle
from helpers import check_close, np32

pytestmark = pytest.mark.gpu


def _caches(B, R, Hq, Hkv, D):
    g = torch.Generator(device="cuda").manual_seed(R + D)
    return [torch.randn(s, generator=g, device="cuda").bfloat16() for s in ((B, Hq, D), (B, R, Hkv, D), (B, R, Hkv, D))]


def _ref(q, k, v, lens, rows):
    """Attention of q over the first lens[b] rows, sequence by sequence."""
    out = []
    for b in rows:
        n = lens[b]
        qf = np.zeros((1, n) + tuple(q.shape[1:]), dtype=np.float32)
        qf[0, n - 1] = np32(q[b])
        out.append(oracle.attn_fwd(qf, np32(k[b:b + 1, :n]), np32(v[b:b + 1, :n]), np.array([0], np.int32),
                                   np.array([n - 1], np.int32), 0)[0][0])
    return np.stack(out)


@pytest.mark.parametrize("ring", [False, True])
@pytest.mark.parametrize("R", [24 * 64, 24 * 64 + 1, 32 * 64, 32 * 64 + 1, 2700])
def test_one_pair_a_cta(ring, R):
    from paper_2608_29539_gb300 import logo as G
    Hq, Hkv, D = 4, 2, 64
    B = G.logo_num_sms()  # two pairs a sequence, two CTAs a multiprocessor
    q, k, v = _caches(B, R, Hq, Hkv, D)
    lens = [64] * B
    for b, n in ((0, R), (7, R - 63), (B // 2, 1000), (B - 1, R)):
        lens[b] = n
    rows = [0, 3, 7, B // 2, B - 1]
    n = torch.tensor(lens, dtype=torch.int32, device="cuda")
    if ring:
        got = G.logo_decode_local_attn(q, k, v, n, R)[rows]
    else:
        p = torch.zeros((B, 1), device="cuda")
        p[rows] = 0.9
        _, _, cu_q, _, ns = G.logo_select(p, G.LOGO_SELECT_THRESHOLD, b_th=0.5)
        got = G.logo_decode_global_sparse_attn(q, k, v, n, cu_q, ns)[:len(rows)]
    torch.cuda.synchronize()
    check_close(np32(got), _ref(q, k, v, lens, rows), "o")
