"""All interleavings of the exchange in which the members of a cluster send each other their rows (attention_kt.cuh), with members that
give up waiting at any moment: no copy may be under way to a member that has left, or out of one, and nobody may wait for good.

A member says that its receive buffer may be written (ready), sends, says that it has received all (received), and leaves.  The rules of
the kernel: send when the other is ready, say "received" when the other's copy has landed, leave when the other has received, all three
also after giving up (its limit there is longer than what a member that has not given up may take, so it does not run out first)."""
import pytest

READY, SENT, RECEIVED, LEFT, GAVE_UP = range(5)
NONE, FLYING, LANDED = range(3)


def explore(send_unready, receive_unlanded):
    """(a copy was under way to or from a member that had left, somebody could not go on)."""
    start = ((0,) * 5, (0,) * 5, (NONE, NONE))               # two members; the copies to each of them
    seen, todo, unsafe, stuck = {start}, [start], False, False
    while todo:
        *members, copies = todo.pop()
        nxt = []

        def member(i, flag, to_other=None):
            m = [list(x) for x in members]
            m[i][flag] = 1
            c = list(copies)
            if to_other is not None:
                c[1 - i] = to_other
            nxt.append((tuple(m[0]), tuple(m[1]), tuple(c)))

        for i in (0, 1):
            me, other = members[i], members[1 - i]
            if copies[i] == FLYING:
                unsafe |= bool(me[LEFT] or other[LEFT])
                nxt.append((members[0], members[1], tuple(LANDED if j == i else c for j, c in enumerate(copies))))
            if me[LEFT]:
                continue
            if not me[GAVE_UP]:
                member(i, GAVE_UP)
            if not me[READY]:
                member(i, READY)
            elif not me[SENT]:
                if other[READY] or (send_unready and me[GAVE_UP]):
                    member(i, SENT, FLYING)
            elif not me[RECEIVED]:
                if copies[i] == LANDED or (receive_unlanded and me[GAVE_UP]):
                    member(i, RECEIVED)
            elif other[RECEIVED]:
                member(i, LEFT)
        stuck |= not nxt and not (members[0][LEFT] and members[1][LEFT])
        todo += [s for s in set(nxt) - seen]
        seen |= set(nxt)
    return unsafe, stuck


def test_exchange_is_safe_whoever_gives_up():
    assert explore(send_unready=False, receive_unlanded=False) == (False, False)


@pytest.mark.parametrize("send_unready", [False, True])
def test_saying_received_without_having_received_is_not(send_unready):
    assert explore(send_unready, receive_unlanded=True)[0]
