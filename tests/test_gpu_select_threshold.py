"""Threshold selection over the whole batch in one launch: every size class and
its edges, one-token sequences, sequences that start inside a thread's tokens,
against the oracle and against the chunked path (sizes beyond the one launch)."""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,T", [
    (1, 1), (32, 1), (1024, 1), (1025, 1), (7, 3), (1, 4096), (2, 2049), (1365, 3), (4, 4096), (3, 5461), (5, 3333),
    (1, 32768), (9, 4001), (2, 65536), (131072, 1), (13, 9999), (4, 50000),
])
@pytest.mark.parametrize("b_th", [-1.0, 0.6, 1.0])
def test_select_threshold_sizes(B, T, b_th):
    from paper_2608_29539_gb300 import logo as L
    g = torch.Generator().manual_seed(B * 31 + T)
    p = torch.rand((B, T), generator=g).mul_(16).round_().div_(16).clamp_(0.01, 0.99).contiguous()  # equal to b_th at times
    p[torch.rand((B, T), generator=g) < 0.05] = 0.6
    zo = oracle.select_threshold(p.numpy(), np.float32(b_th))
    po, co, ro, no = oracle.compact(zo)
    th = torch.tensor([b_th], dtype=torch.float32).cuda()
    for call in (lambda: L.logo_select(p.cuda(), L.LOGO_SELECT_THRESHOLD, b_th=b_th),
                 lambda: L.logo_select_device_threshold(p.cuda(), th),
                 lambda: L.logo_select_noalloc(p.cuda(), L.LOGO_SELECT_THRESHOLD, b_th=b_th)):
        try:
            z, pos, cu_q, row_of, n = call()
        except L.LogoError as e:  # logo_select_noalloc takes up to 4096 sequences
            assert e.code == L.LOGO_ERR_SCRATCH_LIMIT and B > 4096
            continue
        torch.cuda.synchronize()
        assert int(n) == no
        np.testing.assert_array_equal(z.cpu().numpy(), zo)
        np.testing.assert_array_equal(pos.cpu().numpy()[:no], po)
        np.testing.assert_array_equal(cu_q.cpu().numpy(), co)
        np.testing.assert_array_equal(row_of.cpu().numpy(), ro)
