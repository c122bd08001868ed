"""Ordering of the shared slice moments in the actor's front kernel, shown on
the CPU: the kernel's barriers as a graph of what is ordered after what, with
the number of moment buffers read from its source."""
import os
import re

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                   "paper_2609_34325_gb300", "csrc", "actor_front.cu")
TILES = 6


def _ordered_after():
    """Edges event -> events that its barriers and program order put after it,
    for the tiles of one CTA: the issuer and the two halves' epilogue warps."""
    after = {}

    def chain(*events):
        for a, b in zip(events, events[1:]):
            after.setdefault(a, set()).add(b)

    issuer = []
    for n in range(TILES):
        # X's product once the tile before has its QKV; QKV's once X is in place
        # and the tile before has been read out
        issuer += [("issue_x", n), ("issue_q", n)]
        chain(("issue_x", n), ("x_full", n))
        chain(("x_ready", n), ("issue_q", n))
        chain(("issue_q", n), ("q_full", n))
        if n:
            chain(("q_full", n - 1), ("issue_x", n))
            chain(("q_free", n - 1), ("issue_q", n))
    chain(*issuer)
    for h in (0, 1):
        program = []
        for n in range(TILES):
            program += [("write", h, n), ("arrive", h, n), ("read", h, n), ("done", h, n)]
            chain(("x_full", n), ("write", h, n))
            chain(("arrive", h, n), ("x_ready", n))     # a barrier completes after all arrivals
            chain(("x_ready", n), ("read", h, n))
            chain(("q_full", n), ("done", h, n))
            chain(("done", h, n), ("q_free", n))
        chain(*program)
    return after


def _reaches(after, a, b):
    seen, todo = set(), [a]
    while todo:
        e = todo.pop()
        if e == b:
            return True
        if e not in seen:
            seen.add(e)
            todo += after.get(e, ())
    return False


def _unordered(slots):
    """Reads of the other half's moments that a later write to the same buffer
    may overtake."""
    after = _ordered_after()
    return [(h, n, m) for h in (0, 1) for n in range(TILES) for m in range(n + 1, TILES)
            if m % slots == n % slots and
            not _reaches(after, ("read", h, n), ("write", 1 - h, m))]


def test_moments_are_read_before_their_buffer_is_written_again():
    src = open(SRC).read()
    dims = re.search(r"float2 half_moments((?:\[\w+\])+);", src).group(1)
    slots = 1 if dims.count("[") == 2 else int(re.match(r"\[(\d+)\]", dims).group(1))
    uses = re.findall(r"s\.half_moments((?:\[[^\]]+\])+)", src)
    assert len(uses) == 2
    if slots > 1:
        assert slots == 2 and all(u.startswith("[n & 1]") for u in uses)
    assert _unordered(slots) == []


def test_the_model_tells_one_buffer_from_two():
    assert _unordered(1) and not _unordered(2)
