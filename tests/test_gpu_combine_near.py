"""The gate's gradient where the two branches' outputs agree (a transform that is
still the identity, a window that covers the past): dp = sum dO (o~G - o~L) is
taken of each element's difference, so equal branches give exactly zero, with
gains read and without the gains' gradients too."""
import pytest
import torch

from helpers import seeded

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T,H,D", [(300, 1, 64), (500, 5, 64), (400, 32, 128), (130, 48, 128), (77, 64, 128)])
@pytest.mark.parametrize("sums", [False, True])
def test_equal_branches(T, H, D, sums):
    from paper_2608_29539_gb300 import logo as L
    o_l, dO = (seeded((1, T, H, D), H + i).bfloat16().cuda() for i in range(2))
    p = torch.sigmoid(seeded((1, T), H)).cuda()
    gain = 1.0 + 0.1 * seeded((H, D), H + 2).cuda()
    z, pos, _, row_of, n = L.logo_select(p, L.LOGO_SELECT_RATIO, ratio=0.4)
    n = int(n)
    o_c = torch.zeros((T, H, D), dtype=torch.bfloat16, device="cuda")
    o_c[:n] = o_l[0, pos[:n].long()]
    call = L.logo_combine_bwd_gains if sums else L.logo_combine_bwd
    dgate = call(dO, o_l, o_c, p, z, row_of, gain, gain.clone())[2]
    torch.cuda.synchronize()
    assert n > 0 and bool((dgate == 0.0).all()), float(dgate.abs().max())
