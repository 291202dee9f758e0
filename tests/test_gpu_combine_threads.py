"""The combine with gains from several host threads, each with its own head count
and stream: the kernels' launch attributes belong to the process, so no call may
narrow them to its own size."""
import threading

import pytest
import torch

from helpers import seeded

pytestmark = pytest.mark.gpu


def _state(H, D):
    B, T = 1, 64
    o_l, o_c, dO = (seeded((B, T, H, D), H + i).bfloat16().cuda() for i in range(3))
    p = torch.sigmoid(seeded((B, T), H)).cuda()
    gains = [1.0 + 0.1 * seeded((H, D), H + i).cuda() for i in (3, 4)]
    return B, T, o_l, o_c.view(B * T, H, D), dO, p, gains


@pytest.mark.parametrize("heads,D", [((8, 16, 32), 128), ((40, 48, 64), 128), ((8, 32, 64), 64)])
def test_sizes_side_by_side(heads, D):
    from paper_2608_29539_gb300 import logo as L
    states = {}
    for H in heads:
        B, T, o_l, o_c, dO, p, gains = _state(H, D)
        z, _, _, row_of, _ = L.logo_select(p, L.LOGO_SELECT_RATIO, ratio=0.25)
        fwd = lambda a=(o_l, o_c, p, z, row_of, *gains): L.logo_combine(*a)[0]  # noqa: E731
        bwd = lambda a=(dO, o_l, o_c, p, z, row_of, *gains): L.logo_combine_bwd_gains(*a)  # noqa: E731
        want = (fwd(), *bwd())
        states[H] = (fwd, bwd, [want[0], want[1], *want[3:]])
    torch.cuda.synchronize()
    failed, start, done = [], threading.Barrier(len(heads) + 2), threading.Event()
    small = L.Dims(1, 64, heads[0], heads[0], D)

    def ask():  # the size of a workspace, over and over: it looks at the same kernels
        start.wait()
        while not done.is_set():
            L.lib().logo_combine_bwd_workspace_size(small)

    def work(fwd, bwd, want):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                start.wait()
                for _ in range(2000):
                    o = fwd()
                    got = bwd()
                torch.cuda.current_stream().synchronize()
            if not all(torch.equal(a, b) for a, b in zip([o, got[0], *got[2:]], want)):
                failed.append("other results")
        except Exception as e:  # noqa: BLE001
            failed.append(e)

    threads = [threading.Thread(target=work, args=s) for s in states.values()]
    asking = [threading.Thread(target=ask) for _ in range(2)]
    for t in threads + asking:
        t.start()
    for t in threads:
        t.join()
    done.set()
    for t in asking:
        t.join()
    assert not failed, failed
