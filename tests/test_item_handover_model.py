"""The hand-over of work items inside the attention kernel (attn_kernel.cu: the scheduler and item_ready) as a small state
machine, explored over every interleaving and every point at which a bounded wait can run out: all warps see the same items
and all of them end.  (The softmax warps wait for one another once per tile and rely on it.)  The rule the kernel does not
follow, to go by what the slot holds when the wait has run out, is explored too: there warps disagree."""
import pytest

SLOTS, WARPS = 2, 2  # slots of the ring, consumer warps


def explore(items, may_expire, by_slot):
    """Every outcome: a set of tuples, one entry per warp, of the items it saw.  None among them: somebody waits for ever.
    by_slot: a wait that has run out goes by what the slot holds, and a slot is written when the wait for it has run out."""
    # phases completed by full[slot]; releases of every slot; what the slots hold (item or -1); items counted in; no more;
    # has a wait run out; scheduler done; per warp: (next k, items seen, done)
    start = ((0,) * SLOTS, (0,) * SLOTS, (None,) * SLOTS, 0, False, False, False, ((0, (), False),) * WARPS)
    put = lambda t, i, v: t[:i] + (v,) + t[i + 1:]
    seen, todo, outcomes = {start}, [start], set()
    while todo:
        state = todo.pop()
        full, free, holds, pub, closed, expired, over, warps = state
        nxt = []
        if not over:
            slot = pub % SLOTS
            may_write = free[slot] >= WARPS * (pub // SLOTS)
            arrived = put(full, slot, full[slot] + 1)
            last = pub == items or expired or (closed and not by_slot)
            if may_write or (by_slot and (may_expire or expired)):
                nxt.append((arrived, free, put(holds, slot, -1 if last else pub), pub + (not last), closed or last, expired or not may_write, last, warps))
            elif may_expire or expired:
                nxt.append((full, free, holds, pub, True, True, True, warps))
        for w, (k, got, done) in enumerate(warps):
            if done:
                continue
            slot = k % SLOTS
            ready = full[slot] % 2 != (k // SLOTS) % 2  # a wait on the parity of a phase
            if not ready and not (may_expire or expired):
                continue
            more = (holds[slot] is not None and holds[slot] >= 0) if by_slot else pub > k
            item = holds[slot]
            nxt.append((full, put(free, slot, free[slot] + 1) if more else free, holds, pub, closed or not more, expired or not ready, over,
                        put(warps, w, (k + 1, got + (item,), False) if more else (k, got, True))))
        if not nxt:
            outcomes.add(tuple(got for _, got, _ in warps) if over and all(d for _, _, d in warps) else None)
        for s in nxt:
            if s not in seen and all(k <= items + 3 for k, _, _ in s[7]):
                seen.add(s)
                todo.append(s)
    return outcomes


@pytest.mark.parametrize("items", [0, 1, 2, 3, 5])
def test_warps_agree(items):
    assert explore(items, False, False) == {(tuple(range(items)),) * WARPS}  # no timeout: all items, in order
    after = explore(items, True, False)
    assert None not in after
    for a, b in after:
        assert a == b == tuple(range(len(a)))  # a timeout: fewer items, the same ones for every warp


def test_going_by_the_slot_after_a_timeout_lets_them_disagree():
    assert any(x is None or x[0] != x[1] for x in explore(3, True, True))
