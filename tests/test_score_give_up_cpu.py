"""How the scoring kernel's warps leave when a wait has given up: every order of events, on a model of the warps that share
accumulator buffers.

A buffer comes back to its issuing warp over a named barrier, which counts arrivals and does not know whose they are: a warp that arrives
for the next return while this one still lacks the issuing warp completes it in its place, and every later phase lacks an arrival.
So a buffer has two barriers, which its returns take in turn.  The model has one issuing warp, its two buffers and their epilogue
warps; any wait on an mbarrier may give up at any moment, and an MMA may never retire.  All reachable states are visited: none may
be stuck, and no phase of a barrier may count one warp twice."""
import os
import re

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def explore(order, warps, barriers, limit=3_000_000):
    """order: per segment, the buffer of each item as the issuing warp goes through them; barriers: per buffer.
    Returns the number of states, or raises AssertionError with what went wrong."""
    items = [(seg, b) for seg, bufs in enumerate(order) for b in bufs]
    n_buf = 1 + max(b for _, b in items)
    mine = [[seg for seg, x in items if x == b] for b in range(n_buf)]         # the segment of a buffer's r-th item
    team = [(b, w) for b in range(n_buf) for w in range(warps)]
    # issuing warp: (item, step, ok); steps: 0 wait for keys, 1 return barrier, 2 blocked there, 3 issue, 4 done
    # epilogue warp: (returns so far, step, ok); steps: 0 wait for the item, 1 arrive, 2 given up, 3 blocked on the return,
    # 4 blocked on the segment's barrier, 5 done
    # buffer: (landed phases, issued and in flight, items issued, arrivals at each of its barriers)
    start = ((0, 0, True), tuple((0, 0, True) for _ in team), tuple((0, False, 0, (frozenset(),) * barriers) for _ in range(n_buf)), frozenset())

    def buffer_of(iss):
        i = iss[0]
        return items[i][1] if i < len(items) else i - len(items)               # at the end the returns of the last items

    def enter(r, b, ok, seg_bar, who):
        """The state of an epilogue warp that has passed r returns: on to the next item, over the segments' barrier if need be."""
        if r == len(mine[b]) or mine[b][r] != mine[b][r - 1]:
            return (r, 4, ok), seg_bar | {who}
        return (r, 0, ok), seg_bar

    def arrive(bufs, epi, iss, seg_bar, b, n, who):
        """who's arrival at return n of buffer b; releases everyone blocked at that barrier when it is the last."""
        landed, flying, uses, bars = bufs[b]
        x = n % barriers
        assert who not in bars[x], "a return counted one warp twice"
        at = bars[x] | {who}
        if len(at) == warps + 1:
            at = frozenset()
            if iss[1] == 2 and buffer_of(iss) == b and uses % barriers == x:
                iss = (iss[0], 3, iss[2])
            for i, (bb, w) in enumerate(team):
                r, step, ok = epi[i]
                if bb == b and step == 3 and (r + 1) % barriers == x:
                    new, seg_bar = enter(r + 1, b, ok, seg_bar, (bb, w))
                    epi = epi[:i] + (new,) + epi[i + 1:]
        bufs = bufs[:b] + ((landed, flying, uses, bars[:x] + (at,) + bars[x + 1:]),) + bufs[b + 1:]
        return iss, epi, bufs, seg_bar

    def successors(state):
        iss, epi, bufs, seg_bar = state
        out = []
        i, step, ok = iss
        if step == 0:
            if i >= len(items):
                out.append(((i, 4 if i == len(items) + n_buf else 1, ok), epi, bufs, seg_bar))
            else:
                if ok:
                    out.append(((i, 1, True), epi, bufs, seg_bar))     # the keys are there, or have been for an item before
                out.append(((i, 1, False), epi, bufs, seg_bar))        # it has given up, now or before
        elif step == 1:
            b = buffer_of(iss)
            if bufs[b][2] == 0:
                out.append(((i, 3, ok), epi, bufs, seg_bar))
            else:
                out.append(arrive(bufs, epi, (i, 2, ok), seg_bar, b, bufs[b][2], "issuer"))
        elif step == 3:
            b = buffer_of(iss)
            landed, flying, uses, bars = bufs[b]
            if i >= len(items):
                out.append(((i + 1, 0, ok), epi, bufs, seg_bar))
            else:
                for sent in ((True, False) if ok else (False,)):       # an MMA that never retires might as well not have been sent
                    out.append(((i + 1, 0, ok), epi, bufs[:b] + ((landed, flying or sent, uses + 1, bars),) + bufs[b + 1:], seg_bar))
        for b, (landed, flying, uses, bars) in enumerate(bufs):
            if flying:
                out.append((iss, epi, bufs[:b] + ((landed + 1, False, uses, bars),) + bufs[b + 1:], seg_bar))
        for j, (b, w) in enumerate(team):
            r, step, ok = epi[j]
            landed = bufs[b][0]
            put = lambda e: epi[:j] + (e,) + epi[j + 1:]
            if step == 0:
                if ok:
                    assert landed - r in (0, 1), "parities of two phases of an accumulator mixed up"
                    if landed > r:
                        out.append((iss, put((r, 1, True)), bufs, seg_bar))
                out.append((iss, put((r, 2, False)), bufs, seg_bar))
            elif step == 1:
                new, ns = enter(r + 1, b, ok, seg_bar, (b, w))
                out.append(arrive(bufs, put(new), iss, ns, b, r + 1, (b, w)))
            elif step == 2:
                out.append(arrive(bufs, put((r, 3, ok)), iss, seg_bar, b, r + 1, (b, w)))
        if len(seg_bar) == len(team):
            ne = tuple((r, 5 if r == len(mine[b]) else 0, ok) for (b, w), (r, _, ok) in zip(team, epi))
            out.append((iss, ne, bufs, frozenset()))
        return out

    seen, stack = {start}, [start]
    while stack:
        state = stack.pop()
        nxt = successors(state)
        if not nxt:
            assert state[0][1] == 4 and all(e[1] == 5 for e in state[1]), "stuck: %r" % (state,)
        for s in nxt:
            if s not in seen:
                seen.add(s)
                stack.append(s)
        assert len(seen) <= limit, "the model grew beyond what was meant"
    return len(seen)


# every buffer has an item in every segment here, as the segment's barrier is passed behind items
@pytest.mark.parametrize("order,warps", [([[0, 0, 0, 0]], 4), ([[0, 0], [0, 0]], 3), ([[0, 1, 0, 1]], 2), ([[0, 1], [1, 0]], 2),
                                         ([[0, 1, 1, 0, 0, 1]], 1)])
def test_warps_that_give_up_all_leave(order, warps):
    assert explore(order, warps, barriers=2) > 100


@pytest.mark.parametrize("order,warps", [([[0, 0, 0, 0]], 4), ([[0, 1, 0, 1]], 2)])
def test_the_model_sees_returns_taken_for_one_another(order, warps):
    with pytest.raises(AssertionError, match="stuck|counted one warp twice"):
        explore(order, warps, barriers=1)


def test_the_kernel_passes_returns_as_the_model_does():
    """The returns of a buffer at its two barriers in turn: the issuing warp takes one before it issues the next item, an epilogue warp
    arrives with the item read, or waits there if it has given up."""
    with open(os.path.join(ROOT, "paper_2506_08373_b200", "csrc", "score.cu")) as f:
        src = re.sub(r"//[^\n]*", "", f.read())
    first = int(re.search(r"kReturnBarrier = (\d+)", src).group(1))
    others = [int(x) for x in re.findall(r'"bar\.sync (\d+)', src)] + [int(x) + 3 for x in re.findall(r'"r"\((\d+) \+ wg\)', src)]
    assert max(others) < first                                           # the epilogue's barriers among themselves
    kernel = src[src.index("score_kernel(const __grid_constant__"):]
    issuing, epilogue = kernel[:kernel.index("setmaxnreg.inc")], kernel[kernel.index("setmaxnreg.inc"):]
    assert re.search(r"if \(back\) return_sync\(back\);\s*const uint32_t next = back \? back \^ 1 : kReturnBarrier \+ 2 \* buf;", issuing)
    assert "uint32_t ret = kReturnBarrier + 2 * wg;" in epilogue
    take = r"ok = ok && [^;]*mbar_wait_warp\(&t_full\[wg\], ret & 1, abort_flag\)+;\s*if \(!ok\) \{ return_sync\(ret\); ret \^= 1; continue; \}\s*ret \^= 1;"
    assert len(re.findall(take, epilogue)) == 2 and epilogue.count("return_sync(") == 2 and epilogue.count("ret ^= 1;") == 4
    assert set(re.findall(r"return_arrive\([^;]*;", epilogue)) == {"return_arrive(ret ^ 1);"}
