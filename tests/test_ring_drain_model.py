"""A model, run on the CPU, of how the network's kernels leave when a wait runs
out: a loader streams G tiles through a ring of S stages (full and empty
mbarriers, parity waits of at most LIMIT ticks), a consumer frees a stage once
its tile has landed, and the block ends when both have ended.  A copy that lands
later than the consumer's limit must not land after the block has gone: the
loader waits (again with a limit) for its copies when it gives up, and the
consumer, when it is the one that does, for those that may be in flight by then,
since the loader may have issued its last ones and be done."""
import pytest

LIMIT = 50


class _Bar:
    def __init__(self):
        self.phase = 0

    def done(self, parity):  # the phase of that parity has completed
        return (self.phase & 1) != parity


def _run(G, S, late, delay, who):
    """Ticks at which copies land, and the tick at which the block ends; copy
    `late` takes delay ticks, the others two."""
    full, empty = [_Bar() for _ in range(S)], [_Bar() for _ in range(S)]
    flying, landed, now = {}, {}, 0

    def wait(bar, parity):
        for _ in range(LIMIT):
            if bar.done(parity):
                return True
            yield
        return False

    def loader():
        ok, issued = True, 0
        for i in range(G):
            if i >= S:
                ok = yield from wait(empty[i % S], (i // S - 1) & 1)
                if not ok:
                    break
            flying[i] = now + (delay if i == late else 2)
            issued += 1
            yield
        if not ok or who == "loader_at_once":
            for i in range(max(0, issued - S), issued):
                yield from wait(full[i % S], (i // S) & 1)

    def consumer():
        for i in range(G):
            ok = yield from wait(full[i % S], (i // S) & 1)
            if not ok:
                if who == "each":
                    for q in range(i, min(G, i + S)):
                        yield from wait(full[q % S], (q // S) & 1)
                return
            empty[i % S].phase += 1
            yield

    roles, end = [loader(), consumer()], None
    while roles or flying:
        for i in [i for i, t in flying.items() if t <= now]:
            landed[i] = now
            full[i % S].phase += 1
            del flying[i]
        for r in list(roles):
            try:
                next(r)
            except StopIteration:
                roles.remove(r)
        if not roles and end is None:
            end = now
        now += 1
    return landed, end


SHAPES = [(G, S) for S in (2, 4, 5, 8) for G in (1, 2, 5, 17, 26)]


@pytest.mark.parametrize("G,S", SHAPES)
def test_no_copy_lands_after_the_block_has_ended(G, S):
    for late in range(G):
        for delay in (2, LIMIT // 2, LIMIT + 5, 2 * LIMIT - 10):
            landed, end = _run(G, S, late, delay, "each")
            assert max(landed.values()) <= end, (late, delay)
            if delay < LIMIT:
                assert len(landed) == G


@pytest.mark.parametrize("who", ["loader", "loader_at_once"])
def test_a_loader_waiting_alone_is_caught(who):
    """Only when it gives up: the last tiles' copies, all issued, outlive a
    consumer that did.  In any case, as soon as all are issued: its limit runs
    out with the consumer's."""
    def broken(G, S):
        return any(max(landed.values()) > end for late in range(G)
                   for landed, end in [_run(G, S, late, LIMIT + 5, who)])

    assert all(broken(G, S) for G, S in SHAPES)
