"""ContextNorm and fusion with trained gains: token rows shorter than a warp,
rows that share a block, rows of several hundred vectors, fewer tokens than
blocks and many rounds of the copy ring, nothing and everything selected."""
import numpy as np
import pytest
import torch

import oracle
from helpers import check_close, np32, seeded

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,T,H,D,ratio,which", [
    (1, 1, 1, 64, 1.0, "lg"),       # one vector row of 8 in a warp of 32
    (3, 77, 3, 64, 0.3, "lg"),      # 24 vectors, eight rows of threads a block
    (2, 333, 5, 128, 0.5, "l"),     # 80 vectors in 96 threads; no global gain
    (1, 1400, 16, 128, 0.125, "lg"),
    (2, 900, 33, 128, 0.2, "g"),    # 528 vectors: 1024 threads at most
    (1, 130, 64, 128, 0.0, "lg"),
    (1, 65, 128, 64, 1.0, "lg"),
    (1, 20000, 2, 64, 0.1, "lg"),   # more than 64 tokens a warp: the routing's batches
])
def test_combine_gained(B, T, H, D, ratio, which):
    from paper_2608_29539_gb300 import logo as L
    s = 13 * T + H
    p = torch.sigmoid(seeded((B, T), s)).contiguous()
    z, pos, cu_q, row_of, n = L.logo_select(p.cuda(), L.LOGO_SELECT_RATIO, ratio=ratio)
    n = int(n)
    o_l, dO = seeded((B, T, H, D), s + 1, torch.bfloat16), seeded((B, T, H, D), s + 2, torch.bfloat16)
    o_c = seeded((B * T, H, D), s + 3, torch.bfloat16)
    o_c[n:] = float("nan")  # rows that hold nothing
    gl = 1 + 0.1 * seeded((H, D), s + 4) if "l" in which else None
    gg = 1 + 0.1 * seeded((H, D), s + 5) if "g" in which else None
    cu = lambda t: None if t is None else t.cuda()  # noqa: E731
    f32 = lambda t: None if t is None else np32(t)  # noqa: E731
    zn, rown, oc = z.cpu().numpy(), row_of.cpu().numpy(), np32(o_c)[:n]
    o, rl, rg = L.logo_combine(o_l.cuda(), o_c.cuda(), p.cuda(), z, row_of, cu(gl), cu(gg), 1e-6)
    dl, dc, dp, dgl, dgg = L.logo_combine_bwd_gains(dO.cuda(), o_l.cuda(), o_c.cuda(), p.cuda(), z, row_of, cu(gl),
                                                    cu(gg), 1e-6)
    torch.cuda.synchronize()
    ro, rrl, rrg = oracle.combine_fwd(np32(o_l), oc, np32(p), zn, rown, f32(gl), f32(gg), 1e-6)
    check_close(np32(o), ro, "o")
    check_close(np32(rl), rrl, "rstd_l", 0.0, 1e-5, rel=1e-5)
    check_close(np32(rg)[:n], rrg, "rstd_g", 0.0, 1e-5, rel=1e-5)
    rdl, rdc, rdp = oracle.combine_bwd(np32(dO), np32(o_l), oc, np32(p), zn, rown, f32(gl), f32(gg), 1e-6)
    check_close(np32(dl), rdl, "dO_l")
    check_close(np32(dc)[:n], rdc, "dO_c")
    # fp32 sums of H*D products of size ~1: 2^-24 sqrt(H*D) each way, with a wide margin
    check_close(np32(dp), rdp, "dp", 1e-3, 1e-5, rel=1e-5)
    rgl, rgg = oracle.combine_dgain(np32(dO), np32(o_l), oc, np32(p), zn, rown, 1e-6)
    check_close(np32(dgl), rgl, "dgain_l", 1e-2, 1e-5, rel=1e-5)
    check_close(np32(dgg), rgg, "dgain_g", 1e-2, 1e-5, rel=1e-5)
    assert np.isfinite(np32(dgg)).all()
