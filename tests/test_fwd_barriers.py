"""The parity waits of the attention forward, in every interleaving of its
roles.  A parity wait cannot tell a phase from the one two before or after: it
is sound while it is only made with the phase before complete and no later one;
otherwise it passes early, or has been lapped and may never end.  The model has
the two softmax warpgroups (even and odd KV blocks), the P.V issuer and the
epilogue with their barriers; what the epilogue waits on, and how many barriers
the P.V products use in turn, is read from the kernel."""
import os
import re

import pytest

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2608_29539_gb300", "csrc",
                   "attn_fwd.cu")


def explore(items, obufs, own, npv):
    """items: KV blocks of each work item.  own: the epilogue waits on a barrier per O buffer (else on the
    last block's bar_pv_done, of which there are npv).  Returns (unsound waits, dead ends)."""
    first = [sum(items[:i]) for i in range(len(items) + 1)]

    def softmax(par):
        prog = []
        for i, blocks in enumerate(items):
            for g in range(first[i], first[i] + blocks):
                if g % 2 != par:
                    continue
                if g > 0:
                    prog.append(("wait", f"m{1 - par}", (g - 1) // 2))
                prog.append(("arrive", f"m{par}"))
                if g >= 2:
                    prog.append(("wait", f"pv{(g - 2) % npv}", (g - 2) // npv))
                if g >= 1:
                    prog.append(("may wait", f"pv{(g - 1) % npv}", (g - 1) // npv))  # rescaling O
                prog.append(("arrive", f"p{par}"))
            if i > 0:
                prog.append(("wait", "l_empty", i - 1))
            prog.append(("arrive", "l_full"))
        return prog

    issuer, epilogue = [], []
    for i, blocks in enumerate(items):
        ob, use = i % obufs, i // obufs
        for g in range(first[i], first[i] + blocks):
            issuer.append(("wait", f"p{g % 2}", g // 2))
            if g == first[i] and use > 0:
                issuer.append(("wait", f"o_free{ob}", use - 1))
            issuer.append(("arrive", f"pv{g % npv}"))
        issuer.append(("arrive", f"o_full{ob}"))
        last = first[i + 1] - 1
        epilogue += [("wait", "l_full", i), ("arrive", "l_empty"),
                     ("wait", f"o_full{ob}", use) if own else ("wait", f"pv{last % npv}", last // npv),
                     ("arrive", f"o_free{ob}")]
    progs = [softmax(0), softmax(1), issuer, epilogue]
    names = sorted({op[1] for p in progs for op in p})
    at = {n: k for k, n in enumerate(names)}
    arrivals = {"l_full": 2}
    start = ((0,) * 4, (0,) * len(names))
    seen, todo, unsound, dead = {start}, [start], set(), 0
    while todo:
        pcs, count = todo.pop()
        moved = False

        def go(a, after):
            state = (pcs[:a] + (pcs[a] + 1,) + pcs[a + 1:], after)
            if state not in seen:
                seen.add(state)
                todo.append(state)

        for a, prog in enumerate(progs):
            if pcs[a] == len(prog):
                continue
            op = prog[pcs[a]]
            b = at[op[1]]
            if op[0] == "arrive":
                moved = True
                go(a, count[:b] + (count[b] + 1,) + count[b + 1:])
                continue
            phases = count[b] // arrivals.get(op[1], 1)
            if phases not in (op[2], op[2] + 1):
                unsound.add(op[1:])
            if phases % 2 != op[2] % 2 or op[0] == "may wait":
                moved = True
                go(a, count)
        dead += not moved and any(pcs[a] < len(p) for a, p in enumerate(progs))
    return unsound, dead


ITEMS = [[5, 5, 5], [1, 3, 3, 2], [2, 6, 3], [1, 8, 2], [4, 4, 4, 1], [1, 1, 1, 1]]


@pytest.mark.parametrize("items", ITEMS)
@pytest.mark.parametrize("obufs", [1, 2])
def test_waits_are_sound(items, obufs):
    src = open(SRC).read()
    npv = int(re.search(r"uint64_t bar_pv_done\[(\d)\]", src).group(1))
    epilogue = src.split("---- epilogue\n", 1)[1].split("global prep", 1)[0]
    waits = re.findall(r"mbar_wait\w*\(smem_u32\(&bar_(\w+)", epilogue)
    assert waits[0] == "l_full" and waits[1] in ("o_full", "pv_done") and len(waits) == 2
    assert explore(items, obufs, own=waits[1] == "o_full", npv=npv) == (set(), 0)


def test_the_model_shows_a_lapped_wait():
    unsound, dead = explore([5, 5, 5], 2, own=False, npv=4)  # two O buffers, the epilogue on bar_pv_done
    assert unsound and dead
