"""The branch transforms of every row do not depend on how the rows are cut into
sequences: a batch of short ones gives the bits of one long sequence."""
import pytest
import torch

from helpers import seeded

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,T,H,D", [(300, 3, 3, 64), (37, 129, 2, 64), (50, 127, 4, 128), (129, 1, 1, 128), (2, 128, 2, 128)])
@pytest.mark.parametrize("form", ["lp", "so"])
@pytest.mark.parametrize("accumulate", [False, True])
def test_batch_is_one_sequence(B, T, H, D, form, accumulate):
    from paper_2608_29539_gb300 import logo as L
    u, du_g, du0 = (seeded((B, T, H, D), B + i).bfloat16().cuda() for i in range(3))
    if form == "lp":
        a = 0.1 * seeded((H, D, D), T)
        fwd = bwd = {"a": a.bfloat16().cuda()}
    else:
        fwd = {"s": seeded((H, D), T).cuda(), "b": seeded((H, D), T + 1).cuda()}
        bwd = {"s": fwd["s"]}
    got = []
    for b in (B, 1):
        x, g = u.view(b, -1, H, D), du_g.view(b, -1, H, D)
        out = L.logo_branch_transform(x, **fwd)
        grads = L.logo_branch_transform_bwd(x, g, du_l=du0.clone().view(b, -1, H, D), accumulate=accumulate, **bwd)
        got.append([t.reshape(-1) for t in (out, *grads)])
    torch.cuda.synchronize()
    for many, one in zip(*got):
        assert torch.equal(many, one)
