"""Threshold selection on both sides of the sizes where the one launch gives way:
32K tokens of the batch, and the number of chunks from which it does not."""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,T", [(1, 32768), (1, 32769), (32769, 1), (2048, 17), (2049, 17), (1024, 128), (3, 40000), (1, 131073)])
def test_sizes_around_the_limits(B, T):
    from paper_2608_29539_gb300 import logo as L
    p = torch.rand((B, T), generator=torch.Generator().manual_seed(B + T))
    zo = oracle.select_threshold(p.numpy(), np.float32(0.75))
    po, co, ro, no = oracle.compact(zo)
    th = torch.tensor([0.75], device="cuda")
    for z, pos, cu_q, row_of, n in (L.logo_select(p.cuda(), L.LOGO_SELECT_THRESHOLD, b_th=0.75),
                                    L.logo_select_device_threshold(p.cuda(), th)):
        torch.cuda.synchronize()
        assert int(n) == no
        for got, want in ((z, zo), (pos[:no], po), (cu_q, co), (row_of, ro)):
            np.testing.assert_array_equal(got.cpu().numpy(), want)
