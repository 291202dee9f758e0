"""The global decode call serves the packed rows below n_sel_total, also where
that is smaller than what cu_q counts."""
import pytest
import torch

from helpers import seeded

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,L,Hkv,D", [(6, 900, 2, 64), (40, 128, 8, 128)])
@pytest.mark.parametrize("n", [0, 1, 3])
def test_rows_below_n_sel(B, L, Hkv, D, n):
    from paper_2608_29539_gb300 import logo as G
    q, k, v = (seeded(s, B + i).bfloat16().cuda() for i, s in enumerate([(B, Hkv, D)] + 2 * [(B, L, Hkv, D)]))
    lens = torch.full((B,), L, dtype=torch.int32, device="cuda")
    cu_q = torch.div(torch.arange(B + 1, device="cuda") + 1, 2, rounding_mode="floor").int()  # every other sequence
    rows = int(cu_q[-1])
    count = lambda c: torch.tensor([c], dtype=torch.int32, device="cuda")  # noqa: E731
    whole = torch.full((B, Hkv, D), 5.0, dtype=torch.bfloat16, device="cuda")
    some = whole.clone()
    G.logo_decode_global_sparse_attn(q, k, v, lens, cu_q, count(rows), o_c=whole)
    G.logo_decode_global_sparse_attn(q, k, v, lens, cu_q, count(n), o_c=some)
    torch.cuda.synchronize()
    assert bool((some[n:] == 5.0).all()) and bool((whole[rows:] == 5.0).all())
    assert (some[:n].float() - whole[:n].float()).abs().max().item() < 0.05 if n else True
