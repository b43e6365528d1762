"""Order of the shared-memory hand-over of row references in the FP8 P/V kernel, on a model of its roles: which accesses its
barriers order, for any lengths of a CTA's items.  The number of slots is read from the kernel's source."""
import os
import random
import re

import pytest

SOURCE = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2609_04105_b200", "csrc", "attn_fwd_fp8pv.cu")


def _happens_before(stages, writers):
    """stages: of a CTA's items, in order; writers: the teams that write an item's reference.  Returns before(x, y) over the
    events ("write", item, team) and ("read", item).  Edges: the order within a team, the PV issuer and the epilogue, and the
    barriers SMDONE, PFREE, MURDY, OFULL and OFREE."""
    succ, last = {}, {}

    def event(role, name, *after):
        for e in (last.get(role),) + after:
            if e is not None:
                succ.setdefault(e, []).append(name)
        last[role] = name

    n, g, products = len(stages), 0, {}
    steps = []                                                  # (phase, kind, stage of the item, pair), in step order
    for ph in range(n + 1):
        TA, TB = stages[ph] if ph < n else 0, stages[ph - 1] if ph else 0
        for s in range(max(TA, TB)):
            for kind in ((0, 1), (1, 0))[s & 1]:                # 0: first sweep of item ph, 1: second sweep of item ph - 1
                if s < (TB if kind else TA):
                    steps.append((ph, kind, s, g & 1))
                    g += 1
    for ph in range(n + 1):
        for _, kind, s, pair in (x for x in steps if x[0] == ph):
            if not kind:
                continue
            k = ph - 1
            for team in (2 * pair, 2 * pair + 1):
                event(team, ("visit", k, s, team), products.get(pair))              # PFREE: the pair's previous product
            free = ("read", k - 1) if s == 0 and k else None                        # OFREE, signalled after the read
            event("pv", ("product", k, s), ("visit", k, s, 2 * pair), ("visit", k, s, 2 * pair + 1), free)   # SMDONE
            products[pair] = ("product", k, s)
            if s == stages[k] - 1:
                event("epilogue", ("read", k), ("product", k, s))                   # OFULL
        if ph < n:
            for team in range(4):
                event(team, ("arrive", ph, team))
            for team in range(4):                                                   # MURDY: every team
                event(team, ("met", ph, team), *[("arrive", ph, t) for t in range(4)])
                if team in writers:
                    event(team, ("write", ph, team))

    def before(x, y):
        seen, todo = {x}, [x]
        while todo:
            for e in succ.get(todo.pop(), ()):
                if e == y:
                    return True
                if e not in seen:
                    seen.add(e)
                    todo.append(e)
        return False
    return before


def _unordered(stages, slots, writers):
    """Reads that no write of their item precedes, and writes that may overtake a read of the slot's previous item."""
    before = _happens_before(stages, writers)
    bad = [("read", k) for k in range(len(stages)) if not any(before(("write", k, t), ("read", k)) for t in writers)]
    return bad + [("write", k + slots, t) for k in range(len(stages) - slots) for t in writers
                  if not before(("read", k), ("write", k + slots, t))]


def _lengths():
    r = random.Random(3)
    return [[1] * 12, [2] * 12, [1, 2] * 6, [17] + [1] * 9, [1, 1, 3] * 4] + [[r.choice((1, 1, 2, 3, 5)) for _ in range(12)] for _ in range(60)]


def test_reference_slots_are_ordered_between_teams_and_epilogue():
    slots = int(re.search(r"constexpr int kMuSlots = (\d+);", open(SOURCE).read()).group(1))
    for stages in _lengths():
        assert not _unordered(stages, slots, (0, 2)), stages


@pytest.mark.parametrize("slots,writers", [(2, (0,)), (4, (0,)), (2, (0, 2))])
def test_fewer_slots_or_one_writer_are_not_enough(slots, writers):
    """What the model is for: one writing team leaves items of one stage unordered, and two slots may be
    overtaken."""
    assert any(_unordered(stages, slots, writers) for stages in _lengths())
